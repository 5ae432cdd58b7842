"""How the tensor-core GEMM cuts its work at the edges of the rules: three CTAs per two tiles (even and odd tile counts,
ragged last tiles, both sides of the range of tile counts) and clusters of four per tile, at the block sizes where the
stages and the rule change.  Same bound as in test_gpu_linear.py: rounding of K fp32 sums, about sqrt(K) 2^-24."""
import numpy as np
import pytest
import torch

from gpu_util import rel_l2, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    require_gpu()
    from paper_2312_11462_b200 import binding
    binding.csd_set_gemm_path(2)
    yield binding
    binding.csd_set_gemm_path(0)


@pytest.mark.parametrize("m", [1, 5, 6, 8, 9, 10, 11, 17])
@pytest.mark.parametrize("N,K", [(9470, 2048), (9600, 2120), (10600, 2048), (12544, 2056), (12672, 2048), (4096, 1032), (4000, 2048), (3072, 1024)])
def test_shares(b, orc, m, N, K):
    g = torch.Generator(device="cuda")
    g.manual_seed(N + K + m)
    W = (0.05 * torch.randn(N, K, generator=g, device="cuda")).to(torch.bfloat16)
    X = torch.randn(m, K, generator=g, device="cuda")
    Y = b.csd_linear(W, X)
    assert torch.equal(Y, b.csd_linear(W, X))
    ref = orc.linear(orc.blob_to_u16(W).reshape(N, K), X.cpu().numpy())
    assert b.csd_device_status() == 0
    assert rel_l2(Y.cpu().numpy(), ref) < 5e-6
    assert np.abs(Y.cpu().numpy() - ref).max() < 1e-4 * max(1.0, np.abs(ref).max())
