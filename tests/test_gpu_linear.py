"""Parity of the weight-streaming skinny GEMM (csd_linear) with the oracle's contraction."""
import numpy as np
import pytest
import torch

from gpu_util import rel_l2, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=[1, 2, 3], ids=["cuda-core", "tensor-core", "tensor-core-row-ranges"])
def b(request):
    """Every test here runs once per GEMM kernel: 128-bit loads + fp32 FMA, TMA + tcgen05 with equal
    shares of (tile, K block) units, and TMA + tcgen05 with whole output columns per CTA."""
    require_gpu()
    from paper_2312_11462_b200 import binding
    binding.csd_set_gemm_path(request.param)
    yield binding
    binding.csd_set_gemm_path(0)


def case(b, orc, m, N, K, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    W = (0.05 * torch.randn(N, K, generator=g, device="cuda")).to(torch.bfloat16)
    X = torch.randn(m, K, generator=g, device="cuda")
    Y = b.csd_linear(W, X)
    Y2 = b.csd_linear(W, X)                      # split-K partials are summed in a fixed order
    assert torch.equal(Y, Y2)
    ref = orc.linear(orc.blob_to_u16(W).reshape(N, K), X.cpu().numpy())
    got = Y.cpu().numpy()
    # fp32 accumulation of K products of magnitude |w||x|: error ~ sqrt(K) * 2^-24 * |y|
    # (the tensor cores add partial products with a little less care than an fp32 FMA chain)
    assert rel_l2(got, ref) < 5e-6, (m, N, K)
    assert np.abs(got - ref).max() < 1e-4 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("m", [1, 2, 5, 8, 9, 16, 17])
def test_layer_shapes(b, orc, m):
    # the matrix shapes of the small models plus ragged ones (N not a tile multiple, K one
    # partial step, K with a tail slice)
    for N, K in ((768, 768), (2304, 768), (4096, 256), (256, 1024), (64, 64), (1000, 136), (37, 2056), (4099, 520)):
        case(b, orc, m, N, K, seed=N + K + m)


def test_every_block_size(b, orc):
    # all seventeen row counts (every operand padding of the tensor-core kernels: 16, 32, 48, 64 rows of
    # terms) on a shape with several tiles per CTA share and on one with a single short tile
    for m in range(1, 18):
        case(b, orc, m, 3072, 4096, seed=100 + m)
        case(b, orc, m, 200, 1160, seed=200 + m)


@pytest.mark.parametrize("N,K", [(4096, 4096), (12288, 4096), (4096, 11008)])
def test_7b_layer_shapes(b, orc, N, K):
    for m in (5, 17):
        case(b, orc, m, N, K, seed=m)


def test_head_shape_and_uneven_ranges(b, orc):
    # the vocabulary projection (two row ranges per CTA in the row-range kernel) and row counts
    # that leave ranges of unequal length, a K tail and fewer K blocks than a stage holds
    for m, N, K in ((5, 32000, 4096), (3, 20011, 1032), (8, 2371, 4104), (2, 2368, 72)):
        case(b, orc, m, N, K, seed=N + m)


def test_wide_blocks(orc):
    # 18 to 128 rows: the wide-block tensor-core kernel of the prefill.  Each fp32 value enters as two
    # bf16 terms (16 mantissa bits), so the bound is 2^-17-sized, not the 5e-6 of the review kernels.
    require_gpu()
    from paper_2312_11462_b200 import binding as b
    for m, N, K in ((18, 4096, 4096), (64, 12288, 4096), (128, 4096, 11008), (127, 32000, 4096), (33, 4099, 520),
                    (100, 20011, 1032), (128, 2371, 4104)):
        g = torch.Generator(device="cuda")
        g.manual_seed(m + N)
        W = (0.05 * torch.randn(N, K, generator=g, device="cuda")).to(torch.bfloat16)
        X = torch.randn(m, K, generator=g, device="cuda")
        Y = b.csd_linear(W, X)
        assert torch.equal(Y, b.csd_linear(W, X))
        rows = [0, 1, m // 2, m - 2, m - 1]                 # the oracle on a few rows bounds its cost
        ref = orc.linear(orc.blob_to_u16(W).reshape(N, K), X[rows].cpu().numpy())
        got = Y[rows].cpu().numpy()
        assert rel_l2(got, ref) < 3e-5, (m, N, K, rel_l2(got, ref))
        # every row against a float64 product on the GPU side of the harness (torch matmul as the library step)
        full = (X.double() @ W.double().T)
        assert float((Y.double() - full).norm() / full.norm()) < 3e-5
    assert b.csd_device_status() == 0


def test_workspaces_that_hold_anything(orc):
    """The tensor-core kernels count a tile's parts in words of the workspace: what an earlier call on another shape, or
    whoever had the memory before, left there must not matter."""
    require_gpu()
    from paper_2312_11462_b200 import binding as b
    g = torch.Generator(device="cuda")
    g.manual_seed(5)

    def check(m, N, K, ws, bound):
        W = (0.05 * torch.randn(N, K, generator=g, device="cuda")).to(torch.bfloat16)
        X = torch.randn(m, K, generator=g, device="cuda")
        full = X.double() @ W.double().T
        assert float((b.csd_linear(W, X, ws).double() - full).norm() / full.norm()) < bound, (m, N, K)

    for m, N, K in ((18, 12288, 4096), (128, 20000, 1032), (40, 4096, 4096), (9, 12544, 2048), (17, 32000, 768), (1, 12288, 4096)):
        ws = torch.full((b.lib.csd_linear_workspace_bytes(m, N, K),), 0x5a, dtype=torch.uint8, device="cuda")
        check(m, N, K, ws, 3e-5 if m > 17 else 5e-6)
    # a smaller matrix's partial sums lie where a larger one has its tickets
    ws = b.csd_linear_workspace(17, 32000, 4096, "cuda")
    for m, N, K in ((17, 1024, 4096), (17, 32000, 4096), (17, 2048, 4096), (5, 32000, 4096)):
        check(m, N, K, ws, 5e-6)
    assert b.csd_device_status() == 0


@pytest.mark.parametrize("m,N,K", [(18, 1536, 1024), (128, 2304, 1536), (64, 4096, 4096), (33, 4099, 520)])
def test_wide_blocks_into_any_address(m, N, K):
    """A result that starts on a 4-byte boundary only: parts of K as elsewhere, without 16-byte accesses to the result."""
    require_gpu()
    from paper_2312_11462_b200 import binding as b
    g = torch.Generator(device="cuda")
    g.manual_seed(m)
    W = (0.05 * torch.randn(N, K, generator=g, device="cuda")).to(torch.bfloat16)
    X = torch.randn(m, K, generator=g, device="cuda")
    full = X.double() @ W.double().T
    room = torch.full((m * N + 8,), 7.0, device="cuda")
    for off in (0, 1, 2, 3):
        room.fill_(7.0)
        Y = b.csd_linear(W, X, out=room[off:off + m * N].view(m, N))
        assert float((Y.double() - full).norm() / full.norm()) < 3e-5, off
        assert (room[:off] == 7.0).all() and (room[off + m * N:] == 7.0).all()
    assert b.csd_device_status() == 0


@pytest.mark.parametrize("m", [18, 31, 32])
@pytest.mark.parametrize("N,K", [(4096, 4096), (12288, 4096), (2304, 768)])
def test_smallest_wide_blocks_sum_like_fp32(m, N, K):
    """Blocks of up to 32 rows against the fp64 product of the two-term rows themselves: what is left is the fp32 accumulation,
    in chains of 32 tensor-core adds, each truncating up to 2^-23 of the partial sum.  A chain is 512 of the K products, so its
    sum is sqrt(512 / K) of the result and its partial sums 2/3 of that; the losses of a chain point one way and K / 512 chains add
    up like their signs: 32 * 2/3 * 2^-24 * sqrt(512 / K) * sqrt(K / 512) / 2 = 6e-7, half of it on average over a mantissa's range.
    Measured 4.7e-7; with both terms in one chain of 64 adds 1.1e-6."""
    require_gpu()
    from paper_2312_11462_b200 import binding as b
    g = torch.Generator(device="cuda")
    g.manual_seed(m + N)
    W = (0.05 * torch.randn(N, K, generator=g, device="cuda")).to(torch.bfloat16)
    X = torch.randn(m, K, generator=g, device="cuda")
    hi = X.to(torch.bfloat16)
    lo = (X - hi.float()).to(torch.bfloat16)
    full = (hi.double() + lo.double()) @ W.double().T
    assert float((b.csd_linear(W, X).double() - full).norm() / full.norm()) < 7e-7
    assert b.csd_device_status() == 0


@pytest.mark.parametrize("m,N,K", [(18, 64, 16384), (128, 120, 11008), (33, 139, 8192), (100, 57, 20480)])
def test_narrow_wide_blocks(m, N, K):
    """One tile by up to eight parts of K, in scratch of the asked size and with nothing touched behind it."""
    require_gpu()
    from paper_2312_11462_b200 import binding as b
    g = torch.Generator(device="cuda")
    g.manual_seed(N)
    W = (0.05 * torch.randn(N, K, generator=g, device="cuda")).to(torch.bfloat16)
    X = torch.randn(m, K, generator=g, device="cuda")
    full = X.double() @ W.double().T
    n = b.lib.csd_linear_workspace_bytes(m, N, K)
    room = torch.full((n + 4096,), 0x5a, dtype=torch.uint8, device="cuda")
    assert float((b.csd_linear(W, X, room[:n]).double() - full).norm() / full.norm()) < 3e-5
    assert (room[n:] == 0x5a).all()
    assert b.csd_device_status() == 0
