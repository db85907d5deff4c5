"""GPU parity of batched joins whose live pairs all hold one key value each: no digit
to sort by, on the word path's sizes (long arrays), also beside pairs that cannot match and beside one pair of two values."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_21237_gb300 import api
from gpu_util import DEV, assert_pairs_equal, np_of

pytestmark = pytest.mark.gpu

# (R rows, S rows, R's key, S's key) a job
JOBS = {
    "short": [(10, 20_000, 7, 7)],
    "one_job": [(10, 200_000, 7, 7)],
    "single_row": [(1, 130_000, -3, -3)],
    "either_side": [(30, 160_000, 5, 5), (160_000, 30, 1, 1)],
    "with_dead_pairs": [(40, 100_000, 7, 7), (60_000, 60_000, 7, 8), (0, 90_000, 1, 1),
                        (20, 140_000, -(1 << 30), -(1 << 30))],
}


def run(jobs, dtype, ids, second=None):
    kr, ks, ir, is_ = [], [], [], []
    for a, b, x, y in jobs:
        kr.append(torch.full((a,), x, dtype=dtype))
        ks.append(torch.full((b,), y, dtype=dtype))
        ir.append(torch.arange(a, dtype=dtype))
        is_.append(torch.arange(b, dtype=dtype))
    if second is not None:
        ks[0][second] += 1
    if ids == "far":  # no 32-bit window holds them
        ir, is_ = [i << 33 for i in ir], [i << 33 for i in is_]
    r_off = np.concatenate([[0], np.cumsum([j[0] for j in jobs])])
    s_off = np.concatenate([[0], np.cumsum([j[1] for j in jobs])])
    kr, ks, ir, is_ = (torch.cat(x) for x in (kr, ks, ir, is_))
    pairs, off = api.join_batch(r_off.tolist(), s_off.tolist(),
                                *(t.to(DEV) for t in (kr, ir, ks, is_)))
    exp, eoff = oracle.join_batch(r_off, s_off, kr.numpy(), ir.numpy(), ks.numpy(), is_.numpy())
    assert np.array_equal(np_of(off), eoff)
    assert_pairs_equal(pairs, exp)


@pytest.mark.parametrize("jobs", JOBS)
@pytest.mark.parametrize("dtype,ids", [(torch.int32, "near"), (torch.int64, "near"),
                                       (torch.int64, "far")])
def test_pairs_of_one_key(jobs, dtype, ids):
    run(JOBS[jobs], dtype, ids)
    assert api.stats()["radix_passes"] == 0


@pytest.mark.parametrize("dtype", [torch.int32, torch.int64])
def test_one_pair_of_two_values(dtype):
    run(JOBS["either_side"], dtype, "near", second=12_345)
    assert api.stats()["radix_passes"] == 1
