"""Accept calls of a few rows (one kernel, a cluster of CTAs per row) at the edges of its slices:
vocabularies around every cluster size and around the multiples of a warp's stretch, one row and as many
as one wave holds, no drafts to the most, against the oracle."""
import numpy as np
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


@pytest.mark.parametrize("V", [1, 3, 127, 511, 1024, 4095, 4096, 4097, 8193, 32767, 32768, 32772, 65536, 65540, 131072, 131073])
@pytest.mark.parametrize("rows,k", [(1, 0), (1, 1), (3, 4), (9, 2)])
def test_slices(b, orc, V, rows, k):
    t, d, tok = workloads.accept_case(rows, k, V, 0.7, seed=V + rows, device="cuda")
    compare(b, orc, t, d, tok, 1.0, max_flag_frac=0.0)
    compare(b, orc, t, None, tok, 0.8, max_flag_frac=0.0)
    compare(b, orc, t, d, tok, 0.0)


def test_most_drafts_and_one_wave(b, orc):
    t, d, tok = workloads.accept_case(2, 64, 5000, 0.2, seed=4, device="cuda")
    compare(b, orc, t, d, tok, 1.0, max_flag_frac=0.0)
    for rows in (15, 16, 17, 18, 19, 37, 74):                   # up to and past what is resident at once
        t, d, tok = workloads.accept_case(rows, 3, 32000, 0.5, seed=rows, device="cuda")
        compare(b, orc, t, d, tok, 1.0, max_flag_frac=1.0 / rows)       # (16 rows: one within 1e-5 of its threshold)


def test_empty_residual_and_masked_entries(b, orc):
    t, d, tok = workloads.accept_case(4, 2, 9000, 0.5, seed=8, device="cuda")
    # the whole draft law on one entry that the target rules out: the residual is the target law itself
    t2, d2 = t.clone(), torch.full_like(d, float("-inf"))
    tok2 = torch.full_like(tok, 17)
    d2[:, :, 17] = 0.0
    t2[:, :, 17] = float("-inf")
    compare(b, orc, t2, d2, tok2, 1.0)
    # equal laws whose drafts come from elsewhere are accepted; a stretch of masked entries carries no mass
    t3 = t.clone()
    t3[:, :, 100:8990] = float("-inf")
    compare(b, orc, t3, d, tok, 1.0, max_flag_frac=0.0)
