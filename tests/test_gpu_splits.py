"""Splits of the block attention at the cache lengths where their number changes (head dimension 128, more CTAs than
SMs): caches of 4 to 9 key tiles for small and large blocks, and clusters capped at 7, against the oracle."""
import numpy as np
import pytest

import workloads
from workloads import llama_shape
from gpu_util import LOGIT_MAX_ABS, LOGIT_REL_L2, rel_l2, require_gpu, to_dev_i32

pytestmark = pytest.mark.gpu

SHAPE = llama_shape(1, 5120, 40, 512, 500, 600)        # 40 heads: 4 tiles make more CTAs than there are SMs


@pytest.fixture(scope="module")
def b():
    require_gpu()
    from paper_2312_11462_b200 import binding
    return binding


@pytest.fixture(scope="module")
def pair(b, orc):
    blob = workloads.make_weights(SHAPE, seed=44, device="cuda", std=0.03, gain_std=0.2)
    toks = workloads.make_prompt(SHAPE.vocab, SHAPE.max_seq, seed=9)
    om, gm = orc.Model(SHAPE, orc.blob_to_u16(blob)), b.Model(SHAPE, blob)
    om.review_forward(toks[:580], 0)
    gm.csd_prefill(to_dev_i32(toks[:580]), 0)
    return toks, om, gm


@pytest.mark.parametrize("rows", [1, 5, 6, 17])
@pytest.mark.parametrize("cache", [255, 256, 320, 447, 448, 511, 512, 575])
def test_cache_lengths(b, pair, cache, rows):
    toks, om, gm = pair
    blk = toks[cache:cache + rows]
    g, r = gm.csd_review_forward(to_dev_i32(blk), cache).cpu().numpy(), om.review_forward(blk, cache)
    assert b.csd_device_status() == 0
    assert rel_l2(g, r) <= LOGIT_REL_L2, rel_l2(g, r)
    assert np.abs(g - r).max() <= LOGIT_MAX_ABS
