"""GPU parity of budgeted joins of many tiles whose folding route pass meets keys outside
the sampled window at its start, in its middle, at its end or all over, on either side: the
pass ends early and the join runs on separate columns."""
import pytest
import torch

import oracle
from paper_2602_21237_gb300 import api
from gpu_util import DEV, assert_pairs_equal

pytestmark = pytest.mark.gpu

N_R, N_S, STRIDE, SEED = 400_000, 3_000_000, 100, 5
OFF = [(((SEED * m) % (1 << 64)) >> 33) % STRIDE for m in (0x9E3779B97F4A7C15,
                                                           0xBF58476D1CE4E5B9)]


# equal-width ranges; the cut table (many far keys in equal-width ranges would ask for
# ranges over all keys, one of which exceeds the budget)
@pytest.mark.parametrize("at,judge", [(0.0, 0.0), (0.5, 0.0), (0.999, 0.0), (0.0, -1.0),
                                      (0.5, -1.0), (0.999, -1.0), ("many", -1.0)])
@pytest.mark.parametrize("side", [0, 1])
def test_far_key(at, judge, side):
    g = torch.Generator().manual_seed(side)
    keys = [torch.randperm(N_R, generator=g), torch.randint(0, N_R, (N_S,), generator=g)]
    n = keys[side].numel()
    rows = torch.arange(OFF[side] + 1, n, STRIDE)  # none that the sample takes
    rows = rows if at == "many" else rows[int(at * rows.numel())].reshape(1)
    keys[side][rows] = (1 << 50) + torch.arange(rows.numel())
    ids = [torch.arange(N_R), torch.arange(N_S)]
    cols = (keys[0], ids[0], keys[1], ids[1])
    got = api.join_inner(*(t.to(DEV) for t in cols), mem_budget_bytes=32 << 20, router="pla",
                         partitions=64, sample_stride=STRIDE, seed=SEED, radix_judge=judge)
    assert_pairs_equal(got, oracle.join_inner(*(t.numpy() for t in cols)))
