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


@pytest.mark.parametrize("ff", [9608, 9480, 12416], ids=["76-tiles", "75-tiles", "97-tiles"])
def test_gated_pair(orc, ff):
    """Three CTAs per two tiles for gate and up: even and odd tile counts with a ragged last tile, two accumulators parked per
    slot, the activation after the fix-up, on both sides of the sizes where the rule and its constants change."""
    require_gpu()
    import workloads
    from workloads import llama_shape
    from gpu_util import LOGIT_MAX_ABS, LOGIT_REL_L2, to_dev_i32
    from paper_2312_11462_b200 import binding as b
    shape = llama_shape(1, 2048, 16, ff, 600, 160)
    blob = workloads.make_weights(shape, seed=ff, device="cuda", std=0.03, gain_std=0.2)
    om, gm = orc.Model(shape, orc.blob_to_u16(blob)), b.Model(shape, blob)
    toks = workloads.make_prompt(shape.vocab, 160, seed=2)
    pos = 0
    for m in (17, 1, 5, 8, 9, 10, 11, 17, 2, 6):
        g = gm.csd_review_forward(to_dev_i32(toks[pos:pos + m]), pos).cpu().numpy()
        r = om.review_forward(toks[pos:pos + m], pos)
        assert rel_l2(g, r) <= LOGIT_REL_L2, (pos, m, rel_l2(g, r))
        assert np.abs(g - r).max() <= LOGIT_MAX_ABS
        pos += m
    assert b.csd_device_status() == 0
