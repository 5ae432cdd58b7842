"""Wide blocks at the edges of their tiles: prompts of 18 to over 1024 tokens (token tiles of 32 to 256
columns, one to several of them, two passes) and encoder passes, each followed by a review that reads
every cached position, against the oracle's plain forward."""
import numpy as np
import pytest
import torch

import workloads
from workloads import llama_shape, t5_shape
from gpu_util import LOGIT_MAX_ABS, LOGIT_REL_L2, rel_l2, require_gpu, to_dev_i32

pytestmark = pytest.mark.gpu

# matrices just large enough for the wide passes; every one ends inside a row tile
LLAMA = llama_shape(2, 1088, 17, 1416, 500, 1200)
T5 = t5_shape(2, 1, 1088, 17, 64, 1416, 500, 32, 300)


@pytest.fixture(scope="module")
def b():
    require_gpu()
    from paper_2312_11462_b200 import binding
    return binding


@pytest.fixture(scope="module")
def llama_refs(orc):
    """Oracle logits of 3-row reviews behind prompts of the lengths below, from one pass over the text."""
    from paper_2312_11462_b200 import binding as b  # noqa: F401  (GPU tests only)
    blob = workloads.make_weights(LLAMA, seed=41, device="cpu", gain_std=0.2)
    toks = workloads.make_prompt(LLAMA.vocab, LLAMA.max_seq, seed=6)
    om = orc.Model(LLAMA, orc.blob_to_u16(blob))
    refs, pos = {}, 0
    for n in LENGTHS:
        if n > pos:
            om.review_forward(toks[pos:n], pos)
            pos = n
        refs[n] = om.review_forward(toks[n:n + 3], n)     # (rows n .. n+2 are written again by the next stretch)
    return blob, toks, refs


LENGTHS = (18, 31, 32, 33, 64, 127, 128, 129, 255, 256, 257, 300, 513, 700, 1023, 1024, 1025, 1190)


@pytest.mark.parametrize("n", LENGTHS)
def test_prompt_lengths(b, llama_refs, n):
    blob, toks, refs = llama_refs
    m = b.Model(LLAMA, blob.cuda())
    m.csd_prefill(to_dev_i32(toks[:n]), 0)
    g = m.csd_review_forward(to_dev_i32(toks[n:n + 3]), n).cpu().numpy()
    assert b.csd_device_status() == 0
    assert rel_l2(g, refs[n]) <= LOGIT_REL_L2, rel_l2(g, refs[n])
    assert np.abs(g - refs[n]).max() <= LOGIT_MAX_ABS


@pytest.mark.parametrize("n", [33, 300, 1190])
def test_prompts_whose_attention_leaves_fp32_rows(b, llama_refs, n):
    """The CUDA-core attention (the comparison switch; head dimension 32): rotation in the append, its fp32 rows split afterwards."""
    blob, toks, refs = llama_refs
    m = b.Model(LLAMA, blob.cuda())
    try:
        b.csd_set_attention_path(1)
        m.csd_prefill(to_dev_i32(toks[:n]), 0)
        g = m.csd_review_forward(to_dev_i32(toks[n:n + 3]), n).cpu().numpy()
    finally:
        b.csd_set_attention_path(0)
    assert b.csd_device_status() == 0
    assert rel_l2(g, refs[n]) <= LOGIT_REL_L2, rel_l2(g, refs[n])
    assert np.abs(g - refs[n]).max() <= LOGIT_MAX_ABS


@pytest.mark.parametrize("shape,n", [(llama_shape(2, 1088, 34, 1416, 500, 200), 190), (t5_shape(2, 2, 1088, 34, 32, 1416, 500, 32, 150), 150)], ids=["llama", "t5"])
def test_head_dimension_32(b, orc, shape, n):
    blob = workloads.make_weights(shape, seed=44, device="cpu", std=0.01 if shape.arch == 1 else 0.02, gain_std=0.2)
    om, gm = orc.Model(shape, orc.blob_to_u16(blob)), b.Model(shape, blob.cuda())
    toks = workloads.make_prompt(shape.vocab, n + 3, seed=n)
    pos = 0
    if shape.arch == 1:
        om.encoder_forward(toks[:n])
        gm.csd_encoder_forward(to_dev_i32(toks[:n]))
        om.review_forward(toks[:20], 0)                    # (and a prompt of the decoder, through cross-attention)
        gm.csd_prefill(to_dev_i32(toks[:20]), 0)
        pos = 20
    else:
        om.review_forward(toks[:n], 0)
        gm.csd_prefill(to_dev_i32(toks[:n]), 0)
        pos = n
    blk = toks[n:n + 3]
    g, r = gm.csd_review_forward(to_dev_i32(blk), pos).cpu().numpy(), om.review_forward(blk, pos)
    assert b.csd_device_status() == 0
    assert rel_l2(g, r) <= LOGIT_REL_L2, rel_l2(g, r)
    assert np.abs(g - r).max() <= LOGIT_MAX_ABS


@pytest.mark.parametrize("n", [18, 33, 129, 256, 300])
def test_source_lengths(b, orc, n):
    blob = workloads.make_weights(T5, seed=42, device="cpu", std=0.01, gain_std=0.2)
    enc = workloads.make_prompt(T5.vocab, n, seed=n)
    om, gm = orc.Model(T5, orc.blob_to_u16(blob)), b.Model(T5, blob.cuda())
    om.encoder_forward(enc)
    gm.csd_encoder_forward(to_dev_i32(enc))
    blk = np.array([0, 5, 9], dtype=np.int32)
    g, r = gm.csd_review_forward(to_dev_i32(blk), 0).cpu().numpy(), om.review_forward(blk, 0)
    assert b.csd_device_status() == 0
    assert rel_l2(g, r) <= LOGIT_REL_L2, rel_l2(g, r)
    assert np.abs(g - r).max() <= LOGIT_MAX_ABS


@pytest.mark.parametrize("shape", [llama_shape(2, 1024, 16, 1416, 500, 200), llama_shape(1, 1088, 17, 18952, 500, 200)], ids=["d1024", "ff18952"])
def test_models_outside_keep_exact_rows(b, shape):
    """Models outside the sizes of the wide passes: a prompt is what its review-sized blocks are, bit for bit."""
    blob = workloads.make_weights(shape, seed=43, device="cuda", gain_std=0.2)
    toks = to_dev_i32(workloads.make_prompt(shape.vocab, 130, seed=3))
    whole, blocks = b.Model(shape, blob), b.Model(shape, blob)
    whole.csd_prefill(toks[:120].contiguous(), 0)
    for p in range(0, 120, 17):
        blocks.csd_review_forward(toks[p:min(p + 17, 120)].contiguous(), p, append_only=True)
    rows = toks[120:125].contiguous()
    assert torch.equal(whole.csd_review_forward(rows, 120), blocks.csd_review_forward(rows, 120))
    assert b.csd_device_status() == 0


def test_source_longer_than_a_grid_dimension(b):
    """A source of more than 65535 tokens, all equal and without position biases: every position attends to the same value
    whatever the length, so the decoder must see what a short source gives it."""
    shape = t5_shape(1, 1, 64, 2, 32, 128, 64, 8, 65600)
    blob = workloads.make_weights(shape, seed=45, device="cuda", gain_std=0.2)
    at = {name: (off, int(np.prod(shp))) for name, off, shp in workloads.blob_layout(shape)[0]}
    off, count = at["enc.rel_bias"]
    blob[off:off + count] = 0
    m = b.Model(shape, blob)
    out = []
    for n in (24, 65600):
        m.csd_encoder_forward(torch.full((n,), 7, dtype=torch.int32, device="cuda"))
        out.append(m.csd_review_forward(to_dev_i32([1, 2, 3]), 0))
    assert b.csd_device_status() == 0 and torch.isfinite(out[0]).all()
    assert rel_l2(out[1].cpu(), out[0].cpu()) <= 1e-4           # (sums of 65600 fp32 weights: sqrt(65600) 2^-24 each, and K and V entries that round to the neighbour)
