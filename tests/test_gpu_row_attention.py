"""The attention of prompt and source passes at the edges of its 64-row blocks and 64-key tiles, head dimension 128
(test_gpu_wide.py covers 64 with the same lengths): prompts on empty and on filled caches, each followed by a review
that reads every cached position, against the oracle's plain forward."""
import numpy as np
import pytest

import workloads
from workloads import llama_shape
from gpu_util import LOGIT_MAX_ABS, LOGIT_REL_L2, rel_l2, require_gpu, to_dev_i32

pytestmark = pytest.mark.gpu

LLAMA = llama_shape(2, 1152, 9, 1416, 500, 400)


@pytest.fixture(scope="module")
def b():
    require_gpu()
    from paper_2312_11462_b200 import binding
    return binding


@pytest.fixture(scope="module")
def text(orc):
    blob = workloads.make_weights(LLAMA, seed=43, device="cpu", gain_std=0.2)
    toks = workloads.make_prompt(LLAMA.vocab, LLAMA.max_seq, seed=8)
    om = orc.Model(LLAMA, orc.blob_to_u16(blob))
    om.review_forward(toks[:390], 0)
    return blob, toks, om


@pytest.mark.parametrize("parts", [(18,), (63,), (64,), (65,), (128,), (129,), (193,), (64, 64), (30, 99), (130, 18), (255, 66)])
def test_prompt_parts(b, text, parts):
    blob, toks, om = text
    m, n = b.Model(LLAMA, blob.cuda()), 0
    for p in parts:
        m.csd_prefill(to_dev_i32(toks[n:n + p]), n)
        n += p
    g, r = m.csd_review_forward(to_dev_i32(toks[n:n + 3]), n).cpu().numpy(), om.review_forward(toks[n:n + 3], n)
    assert b.csd_device_status() == 0
    assert rel_l2(g, r) <= LOGIT_REL_L2, rel_l2(g, r)
    assert np.abs(g - r).max() <= LOGIT_MAX_ABS
