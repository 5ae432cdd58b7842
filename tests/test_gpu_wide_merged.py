"""Tiles of up to 128 tokens, whose MMAs multiply both terms of the rows at once: widths of 64 to 256 columns and token counts
that end inside a tile, for a single matrix and for both forms of the gated pair (up to 64 tokens, beyond)."""
import numpy as np
import pytest
import torch

import workloads
from workloads import llama_shape
from gpu_util import LOGIT_MAX_ABS, LOGIT_REL_L2, rel_l2, require_gpu, to_dev_i32

pytestmark = pytest.mark.gpu

SHAPE = llama_shape(2, 1088, 17, 1416, 500, 140)
LENGTHS = (40, 63, 65, 96, 97, 112)


@pytest.fixture(scope="module")
def b():
    require_gpu()
    from paper_2312_11462_b200 import binding
    return binding


@pytest.fixture(scope="module")
def refs(orc):
    blob = workloads.make_weights(SHAPE, seed=71, device="cpu", gain_std=0.2)
    toks = workloads.make_prompt(SHAPE.vocab, SHAPE.max_seq, seed=9)
    om = orc.Model(SHAPE, orc.blob_to_u16(blob))
    out, pos = {}, 0
    for n in LENGTHS:
        om.review_forward(toks[pos:n], pos)
        pos = n
        out[n] = om.review_forward(toks[n:n + 3], n)
    return blob, toks, out


@pytest.mark.parametrize("n", LENGTHS)
def test_prompts(b, refs, n):
    blob, toks, out = refs
    m = b.Model(SHAPE, blob.cuda())
    m.csd_prefill(to_dev_i32(toks[:n]), 0)
    g = m.csd_review_forward(to_dev_i32(toks[n:n + 3]), n).cpu().numpy()
    assert b.csd_device_status() == 0
    assert rel_l2(g, out[n]) <= LOGIT_REL_L2, rel_l2(g, out[n])
    assert np.abs(g - out[n]).max() <= LOGIT_MAX_ABS


@pytest.mark.parametrize("m", [33, 64, 65, 96, 97, 128])
@pytest.mark.parametrize("N,K", [(4096, 4096), (12288, 4096), (2371, 4104)])
def test_terms_sum_like_fp32(b, m, N, K):
    """Against the fp64 product of the two-term rows themselves.  What is left is the fp32 accumulation of the high terms, in chains
    of 32 tensor-core adds: 32 * 2/3 * 2^-24 * sqrt(512 / K) * sqrt(K / 512) / 2 = 6e-7 as for blocks of up to 32 rows
    (test_gpu_linear.py); both terms in one chain of 64 adds leave 1.1e-6."""
    g = torch.Generator(device="cuda")
    g.manual_seed(m + N)
    W = (0.05 * torch.randn(N, K, generator=g, device="cuda")).to(torch.bfloat16)
    X = torch.randn(m, K, generator=g, device="cuda")
    hi = X.to(torch.bfloat16)
    lo = (X - hi.float()).to(torch.bfloat16)
    full = (hi.double() + lo.double()) @ W.double().T
    err = float((b.csd_linear(W, X).double() - full).norm() / full.norm())
    print("rel", m, N, K, err, float((b.csd_linear(W, X).double() - X.double() @ W.double().T).norm() / full.norm()))
    assert err < 7e-7, err
    assert b.csd_device_status() == 0
