"""Accept calls that take the passes (more rows or longer vectors than the one-kernel form holds): sizes
at the edges of their pieces (8192 logits) and, beyond 65536, of the resample chunks (1024), the most drafts, scratch
that holds anything, masked and empty laws, and calls that follow one another on a stream, against the oracle."""
import pytest
import torch

import workloads
from gpu_util import require_gpu
from test_gpu_accept import compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    require_gpu()
    from paper_2312_11462_b200 import binding
    return binding


@pytest.mark.parametrize("V", [1, 5, 511, 513, 2049, 8191, 8193, 16385, 65537])
@pytest.mark.parametrize("rows,k", [(200, 1), (150, 4), (160, 0)])
def test_edges(b, orc, V, rows, k):
    t, d, tok = workloads.accept_case(rows, k, V, 0.7, seed=V + rows, device="cuda")
    compare(b, orc, t, d, tok, 1.0)
    compare(b, orc, t, None, tok, 0.8)
    compare(b, orc, t, d, tok, 0.0)


def test_most_drafts_and_long_vectors(b, orc):
    t, d, tok = workloads.accept_case(40, 64, 9001, 0.2, seed=4, device="cuda")
    compare(b, orc, t, d, tok, 1.0)
    t, d, tok = workloads.accept_case(1, 3, 200001, 0.2, seed=5, device="cuda")
    compare(b, orc, t, d, tok, 1.0, max_flag_frac=0.0)
    on = (torch.arange(40 * 64, device="cuda").reshape(40, 64) % 5 == 0).to(torch.int32)
    t, d, tok = workloads.accept_case(40, 64, 9001, 0.1, seed=6, device="cuda")
    compare(b, orc, t, d, tok, 1.3, lenience=2.0, onehot=on)


def test_empty_residual_and_masked_entries(b, orc):
    t, d, tok = workloads.accept_case(170, 2, 9000, 0.5, seed=8, device="cuda")
    t2, d2 = t.clone(), torch.full_like(d, float("-inf"))
    tok2 = torch.full_like(tok, 17)
    d2[:, :, 17] = 0.0                                          # the whole draft law on an entry that the target rules out
    t2[:, :, 17] = float("-inf")
    compare(b, orc, t2, d2, tok2, 1.0)
    t3 = t.clone()
    t3[:, :, 100:8990] = float("-inf")
    compare(b, orc, t3, d, tok, 1.0)


def test_scratch_that_holds_anything_and_calls_in_a_row(b):
    t, d, tok = workloads.accept_case(64, 5, 20000, 0.5, seed=9, device="cuda")
    want = b.csd_spec_accept(t, d, tok, 1.0, seed=3)
    ws = b.csd_spec_accept_workspace(64, 5, 20000, "cuda")
    outs = [tuple(torch.full((64,), -7, dtype=torch.int32, device="cuda") for _ in range(2)) for _ in range(12)]
    for i, out in enumerate(outs):
        if i % 3 == 0:
            ws.view(torch.uint8).fill_(0xff if i % 2 else 0x5a)
        b.csd_spec_accept(t, d, tok, 1.0, seed=3, workspace=ws, out=out)
    for out in outs:
        assert torch.equal(out[0], want[0]) and torch.equal(out[1], want[1])
    bad = tok.clone()
    bad[7, 2] = 20000
    b.csd_spec_accept(t, d, bad, 1.0, seed=3)
    assert b.csd_device_status() == 6                           # a token outside the vocabulary is recorded


@pytest.mark.parametrize("V", [65537, 70001, 131584])
@pytest.mark.parametrize("sigma", [0.0, 1e-5, 1e-3, 0.03, 0.5])
def test_laws_that_nearly_agree(b, orc, V, sigma):
    """Long vocabularies: the entries the residual keeps are told before the normalisers are known but where the laws nearly agree
    (within 5e-5 of their logarithms); those are listed, six a chunk of 1024, and chunks with more are formed anew.  Two entries
    of each draft law are swapped, the drafted one gaining, so that it is refused while all others agree up to sigma."""
    rows, k = 20, 2
    t, _, _ = workloads.accept_case(rows, k, V, 0.5, seed=V, device="cuda")
    g = torch.Generator(device="cuda")
    g.manual_seed(V)
    d = t[:, :k].clone()
    top = d.argmax(-1, keepdim=True)
    low = torch.randint(0, V, (rows, k, 1), generator=g, device="cuda")
    low = torch.where(low == top, (low + 1) % V, low)
    hi_v, lo_v = d.gather(-1, top), d.gather(-1, low)
    d.scatter_(-1, top, lo_v).scatter_(-1, low, hi_v)
    d = (d + sigma * torch.randn(d.shape, generator=g, device="cuda")).contiguous()
    compare(b, orc, t, d, low[..., 0].to(torch.int32).contiguous(), 1.0)
    compare(b, orc, t, d, low[..., 0].to(torch.int32).contiguous(), 0.6)
