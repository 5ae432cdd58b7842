"""Accept calls over vocabularies beyond 65536, whose resample tells before the normalisers are known which entries the residual keeps
and lists up to six undecided ones a chunk (1024 logits; 4096 where the scratch is small), against the oracle."""
import numpy as np
import pytest
import torch

import workloads
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    require_gpu()
    from paper_2312_11462_b200 import binding
    return binding


def workspaces(b, rows, k, V):
    """Scratch as the query function gives it, and the least that is accepted (chunks four times as long)."""
    full = b.lib.csd_spec_accept_workspace_bytes(rows, k, V)
    short = full - 24 * rows * (-(-V // 512) - -(-V // 2048)) + 1024        # (1024: the parts start on 256-byte boundaries)
    return [torch.full((n,), 0x5a, dtype=torch.uint8, device="cuda") for n in (full, short)]


def compare(b, orc, t, d, tok, temperature=1.0, **kw):
    rows, k1, V = t.shape
    n_ref, o_ref, flags = orc.spec_accept(t.cpu().numpy(), d.cpu().numpy(), tok.cpu().numpy(), temperature, 1.0, 7, 3,
                                          onehot=None if "onehot" not in kw else kw["onehot"].cpu().numpy())
    ok = flags == 0
    assert (~ok).mean() <= 0.02
    for ws in workspaces(b, rows, k1 - 1, V):
        n, o = b.csd_spec_accept(t, d, tok, temperature, 1.0, 7, 3, workspace=ws, **kw)
        assert b.csd_device_status() == 0
        assert (n.cpu().numpy()[ok] == n_ref[ok]).all() and (o.cpu().numpy()[ok] == o_ref[ok]).all()
    return n_ref, o_ref


def laws_that_agree_but_for_one_entry(rows, V, each, seed):
    """Both laws on each(chunk) entries of every chunk of 1024, at random places and alike but for one: the draft law's weight on
    that entry, the drafted one, is 5 larger in logarithm, 2e-5 of the whole.  So it is refused nearly always, and all others,
    undecided, carry the residual."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    chunks = V // 1024
    order = torch.rand(rows, chunks, 1024, generator=g, device="cuda").argsort(-1).argsort(-1)
    keep = torch.tensor([each(c) for c in range(chunks)], device="cuda")[None, :, None]
    t = torch.where(order < keep, 2.0 * torch.randn(rows, chunks, 1024, generator=g, device="cuda"), float("-inf")).reshape(rows, V)
    x = torch.randint(0, V, (rows, 1), generator=g, device="cuda")
    t.scatter_(1, x, float("-inf"))
    t.scatter_(1, x, (torch.logsumexp(t.double(), 1, keepdim=True) + np.log(2e-5 / (np.exp(5.0) - 1))).float())
    d = t.scatter_add(1, x, torch.full_like(x, 5.0, dtype=torch.float32))
    return torch.stack([t, t], 1).contiguous(), d[:, None].contiguous(), x.to(torch.int32)


@pytest.mark.parametrize("rows,each", [(40, lambda c: 4 + c % 5), (40, lambda c: c % 3), (40, lambda c: 1024), (40, lambda c: (0, 3, 7)[c % 3]),
                                       (300, lambda c: 1024)],
                         ids=["around-a-full-list", "few", "all", "mixed", "all, many waves of blocks"])
def test_undecided_entries(b, orc, rows, each):
    t, d, tok = laws_that_agree_but_for_one_entry(rows, 66560, each, seed=3)
    n, o = compare(b, orc, t, d, tok)
    assert n.mean() < 0.2 and len(set(o // 1024)) > 15           # the residual is drawn from all over the vocabulary


def test_full_lists_do_not_stand_in_line(b):
    """Chunks with full lists are formed anew by as many CTAs as fit, so such a call takes at most one more pass over the laws it has been
    through twice.  (By one warp a row it took twelve to twenty times as long.)"""
    V, rows = 66560, 20
    near = laws_that_agree_but_for_one_entry(rows, V, lambda c: 1024, seed=4)
    far = (near[0], near[0][:, :1] + 0.5 * torch.randn(rows, 1, V, device="cuda"), near[2])
    out = tuple(torch.empty(rows, dtype=torch.int32, device="cuda") for _ in range(2))
    ws = b.csd_spec_accept_workspace(rows, 1, V, "cuda")

    def us(t, d, tok):
        best = []
        for _ in range(7):
            start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            start.record()
            for _ in range(20):
                b.csd_spec_accept(t, d, tok, 1.0, seed=7, step=3, workspace=ws, out=out)
            end.record()
            end.synchronize()
            best.append(start.elapsed_time(end) / 20 * 1e3)
        return sorted(best)[3]

    a, c = us(*near), us(*far)
    print("us", a, c)
    assert a < 3 * c, (a, c)


@pytest.mark.parametrize("V", [65537, 66559, 66560, 66561, 69631, 69632, 69633])
@pytest.mark.parametrize("rows,k", [(150, 1), (1, 16)])
def test_chunk_edges(b, orc, V, rows, k):
    """One more and one less logit than whole chunks of 1024 and 4096; many rows, and so few that blocks are smaller."""
    t, d, tok = workloads.accept_case(rows, k, V, 0.5, seed=V + rows, device="cuda")
    compare(b, orc, t, d, tok)


def masked(law, rows, k, V):
    """A block whose target law, draft law or both leave entries out."""
    t, d, tok = workloads.accept_case(rows, k, V, 0.5, seed=V, device="cuda")
    every = torch.arange(V, device="cuda")
    x = torch.full_like(tok, V - 3)
    if law == "target":
        t[:, :, every % 3 != 0] = float("-inf")
    elif law == "draft":
        d[:, :, every % 3 != 0] = float("-inf")
        tok = tok // 3 * 3
    elif law == "both":
        t[:, :, every % 2 == 0] = float("-inf")
        d[:, :, every % 3 != 0] = float("-inf")
        tok = tok // 3 * 3
    elif law == "apart":                                     # no entry in common: all of the target's stay
        t[:, :, every % 2 == 0] = float("-inf")
        d[:, :, every % 2 == 1] = float("-inf")
        tok = tok // 2 * 2
    elif law == "one entry":                                 # the whole draft law on an entry that the target has, or has not
        d.fill_(float("-inf"))
        d.scatter_(2, x[..., None].long(), 0.0)
        t[::2, :, V - 3] = float("-inf")
        tok = x
    elif law == "chunks":                                    # whole chunks without an entry, the ends among them
        t[:, :, (every // 4096) % 3 == 0] = float("-inf")
        t[:, :, 65000:] = float("-inf")
    elif law == "near":                                      # laws that nearly agree on half of the vocabulary, which both leave otherwise out
        d = t[:, :k] + 1e-6 * torch.randn(d.shape, device="cuda")
        low = t[:, :k].argmin(-1, keepdim=True)
        d.scatter_add_(2, low, torch.full_like(low, 4.0, dtype=torch.float32))
        gone = (every % 2 == 0)[None, None].expand(rows, k, V) & (every[None, None] != low)
        t[:, :k][gone], d[gone] = float("-inf"), float("-inf")
        tok = low[..., 0].to(torch.int32)
    return t.contiguous(), d.contiguous(), tok.contiguous()


@pytest.mark.parametrize("V", [70001, 131584])
@pytest.mark.parametrize("law", ["target", "draft", "both", "apart", "one entry", "chunks", "near"])
def test_masked_laws(b, orc, law, V):
    rows, k = 12, 2
    t, d, tok = masked(law, rows, k, V)
    compare(b, orc, t, d, tok)
    compare(b, orc, t, d, tok, 0.7)
    # some positions drafted by a statistical model: point masses beside laws
    on = (torch.arange(rows * k, device="cuda").reshape(rows, k) % 3 == 0).to(torch.int32)
    compare(b, orc, t, d, tok, onehot=on)
