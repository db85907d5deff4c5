"""GPU parity of budgeted joins over equal-width ranges of a sampled key range when a
key above the sample's largest lies beyond the equal-width range of that one: it is
routed with the largest sampled keys and must not meet theirs."""
import pytest
import torch

import oracle
from paper_2602_21237_gb300 import api
from gpu_util import DEV, assert_pairs_equal

pytestmark = pytest.mark.gpu

N, STRIDE, SEED = 200_000, 10, 5
OFF = (((SEED * 0x9E3779B97F4A7C15) % (1 << 64)) >> 33) % STRIDE   # first sampled row of R
OFF_S = (((SEED * 0xBF58476D1CE4E5B9) % (1 << 64)) >> 33) % STRIDE


# 64 ranges of 4096 keys: the sampled keys end in [196608, 200704); 201500 is four
# times 1024 and 796 keys into that range, 197404 is 796
@pytest.mark.parametrize("far", [200_703, 200_704, 201_500, 250_000, 1 << 50])
@pytest.mark.parametrize("both", [False, True])
@pytest.mark.parametrize("ids", ["positions", "full"])  # folded rows, separate columns
def test_key_above_the_sampled_range(far, both, ids):
    g = torch.Generator().manual_seed(19)
    kr = torch.randperm(N, generator=g)
    ks = torch.randint(0, N, (2 * N,), generator=g)
    ks[OFF_S + 1 + 500 * STRIDE] = far
    if both:
        kr[OFF + 1 + 700 * STRIDE] = far
    ir, is_ = torch.arange(N), torch.arange(2 * N)
    if ids == "full":
        ir, is_ = (torch.randint(-(1 << 62), 1 << 62, t.shape, generator=g) for t in (ir, is_))
    got = api.join_inner(*(t.to(DEV) for t in (kr, ir, ks, is_)), mem_budget_bytes=6 << 20,
                         router="pla", partitions=64, sample_stride=STRIDE, seed=SEED)
    assert api.stats()["learned"] >= 100  # equal-width ranges
    assert_pairs_equal(got, oracle.join_inner(kr.numpy(), ir.numpy(), ks.numpy(), is_.numpy()))
