"""The words in which GEMMs count a tile's parts: a launch that has given up waiting (its status says so) leaves any count there, and
the next forward must not take it for its own.  Counts are left behind by hand; results are those of a handle without them."""
import pytest
import torch

import workloads
from workloads import llama_shape, t5_shape
from gpu_util import require_gpu, to_dev_i32

pytestmark = pytest.mark.gpu

LLAMA, T5 = llama_shape(2, 4096, 32, 1416, 500, 420), t5_shape(2, 2, 1088, 17, 64, 1416, 500, 96, 320)


@pytest.fixture(scope="module")
def b():
    require_gpu()
    from paper_2312_11462_b200 import binding
    return binding


def ticket_words(b, monkeypatch, shape, blob):
    """First and number of the words: of a workspace, creation zeroes them alone (and writes some tables)."""
    with monkeypatch.context() as mp:
        mp.setattr(b, "_ws", lambda nbytes, device: torch.full((nbytes,), 0xa5, dtype=torch.uint8, device=device))
        zero = b.Model(shape, blob).workspace.view(torch.int32) == 0
    edge = torch.diff(zero.to(torch.int8), prepend=torch.zeros(1, dtype=torch.int8, device="cuda"), append=torch.zeros(1, dtype=torch.int8, device="cuda"))
    first, end = (edge == 1).nonzero()[:, 0], (edge == -1).nonzero()[:, 0]
    at = int((end - first).argmax())
    widest = max(3 * shape.d_inner, shape.d_model, shape.d_ff, shape.vocab)
    assert int(end[at] - first[at]) >= widest + 8                  # (a word per group of rows of the CUDA-core kernel)
    return int(first[at]), 8 * -(-widest // 128)                   # those that waiting kernels count in: eight per 128 outputs


def prompts(m, toks, dirty):
    out, pos = [], 0
    for n in (20, 60, 330):                                        # K parts; shares of q|k|v; two token tiles
        dirty()
        m.csd_prefill(to_dev_i32(toks[pos:n]), pos)
        dirty()
        out.append(m.csd_review_forward(to_dev_i32(toks[n:n + 5]), n))
        pos = n
    return out


def source(m, toks, dirty):
    out = []
    for n in (40, 300):
        dirty()
        m.csd_encoder_forward(to_dev_i32(toks[:n]))
        for r in (4, 17):
            dirty()
            out.append(m.csd_review_forward(to_dev_i32(toks[:r]), 0))
    return out


def blocks(m, toks, dirty):
    out = []
    for r in (1, 5, 8, 12, 17):                                    # rows gathered by the first projection, and embedded first
        dirty()
        out.append(m.csd_review_forward(to_dev_i32(toks[:r]), 0))
    return out


@pytest.mark.parametrize("shape,calls", [(LLAMA, prompts), (T5, source), (workloads.SHAPES["draft68m"], blocks), (workloads.SHAPES["tiny_target"], blocks)],
                         ids=["prompts", "source", "draft", "tiny"])
def test_counts_left_behind(b, monkeypatch, shape, calls):
    blob = workloads.make_weights(shape, seed=5, device="cuda")
    at, n = ticket_words(b, monkeypatch, shape, blob)
    toks = workloads.make_prompt(shape.vocab, 400, seed=3)
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    clean, marked = b.Model(shape, blob), b.Model(shape, blob)
    words = marked.workspace.view(torch.int32)[at:at + n]
    want = calls(clean, toks, lambda: None)
    got = calls(marked, toks, lambda: words.copy_(torch.randint(1, 9, (n,), generator=g, device="cuda", dtype=torch.int32)))
    assert b.csd_device_status() == 0
    for x, y in zip(want, got):
        assert torch.equal(x, y)
    assert not words.any()
