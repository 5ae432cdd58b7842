"""Accept calls over vocabularies beyond 65536, whose resample tells before the normalisers are known which entries the residual keeps
and lists up to six undecided ones a chunk (1024 logits; 4096 where the scratch is small), against the oracle."""
import numpy as np
import pytest
import torch

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
