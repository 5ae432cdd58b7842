"""The row kernel (small matrices, blocks of up to 8 rows) at the edges of its steps: K around multiples of
256 and at its most, N that ends inside a warp's rows and around the counts where a warp takes more rows,
every block size, the norm, the gated pair and the residual add through whole forwards."""
import numpy as np
import pytest
import torch

import workloads
from workloads import llama_shape, t5_shape
from gpu_util import LOGIT_MAX_ABS, LOGIT_REL_L2, rel_l2, require_gpu, to_dev_i32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    require_gpu()
    from paper_2312_11462_b200 import binding
    return binding


@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 6, 7, 8, 9])
def test_shapes(b, m):
    for N, K in ((1, 8), (7, 64), (2368, 256), (2369, 264), (2370, 768), (9475, 520), (33, 776), (769, 3072), (50, 3080)):
        g = torch.Generator(device="cuda")
        g.manual_seed(m + N + K)
        W = (0.05 * torch.randn(N, K, generator=g, device="cuda")).to(torch.bfloat16)
        X = torch.randn(m, K, generator=g, device="cuda")
        want = X.double() @ W.double().T
        got = b.csd_linear(W, X)
        # K fp32 products in up to 8 K / 256 adds a lane and a tree over the lanes: error ~ sqrt(K) 2^-24, bound as for the other kernels
        assert float((got.double() - want).norm() / want.norm()) < 5e-6, (m, N, K)
        assert torch.equal(got, b.csd_linear(W, X))
    assert b.csd_device_status() == 0


@pytest.mark.parametrize("m", [1, 5, 6, 8])
def test_rounding_of_long_sums(b, m):
    """K = 3072: 96 products a lane.  In two chains of 48 adds, partial sums of sqrt(j) terms round to 2^-25 of themselves, rms
    sqrt(2 / 3): sqrt(48 / 2) 2^-25 sqrt(2 / 3) = 1.2e-7 of the result, the tree over lanes and columns under 0.5e-7 more; in one chain
    1.7e-7 and more."""
    g = torch.Generator(device="cuda")
    g.manual_seed(m)
    W = (0.05 * torch.randn(768, 3072, generator=g, device="cuda")).to(torch.bfloat16)
    X = torch.randn(m, 3072, generator=g, device="cuda")
    want = X.double() @ W.double().T
    assert float((b.csd_linear(W, X).double() - want).norm() / want.norm()) < 1.65e-7
    assert b.csd_device_status() == 0


@pytest.mark.parametrize("shape", [llama_shape(2, 768, 12, 3072, 3001, 96), llama_shape(1, 512, 8, 776, 777, 96), t5_shape(1, 2, 512, 8, 64, 1000, 700, 96, 40)],
                         ids=["d768", "d512", "t5-d512"])
def test_forwards(b, orc, shape):
    blob = workloads.make_weights(shape, seed=51, device="cpu", std=0.03 if shape.arch == 0 else 0.01, gain_std=0.2)
    om, gm = orc.Model(shape, orc.blob_to_u16(blob)), b.Model(shape, blob.cuda())
    if shape.arch == 1:
        enc = workloads.make_prompt(shape.vocab, 37, seed=2)
        om.encoder_forward(enc)
        gm.csd_encoder_forward(to_dev_i32(enc))
    toks = workloads.make_prompt(shape.vocab, 96, seed=3)
    pos = 0
    for m in (17, 1, 2, 3, 4, 5, 6, 7, 8, 9, 12, 1):
        g = gm.csd_review_forward(to_dev_i32(toks[pos:pos + m]), pos).cpu().numpy()
        r = om.review_forward(toks[pos:pos + m], pos)
        assert rel_l2(g, r) <= LOGIT_REL_L2, (pos, m, rel_l2(g, r))
        assert np.abs(g - r).max() <= LOGIT_MAX_ABS
        pos += m
    assert b.csd_device_status() == 0
