"""GPU parity of budgeted joins whose key range is read off a sample when the keys lie
at an end of int64: a key of the other end that the sample misses keeps its place in
the order, in regions sized by the sample and by a route histogram."""
import pytest
import torch

import oracle
from paper_2602_21237_gb300 import api
from gpu_util import DEV, assert_pairs_equal

pytestmark = pytest.mark.gpu

INFO = torch.iinfo(torch.int64)
STRIDE, SEED = 10, 5
OFF = (((SEED * 0x9E3779B97F4A7C15) % (1 << 64)) >> 33) % STRIDE   # first sampled row of R
OFF_S = (((SEED * 0xBF58476D1CE4E5B9) % (1 << 64)) >> 33) % STRIDE


# equal-width ranges; the cut table, with regions from the sample and from a histogram
@pytest.mark.parametrize("judge,exact", [(0.0, False), (-1.0, False), (-1.0, True)])
@pytest.mark.parametrize("gap", [0, 700, 1 << 40])  # between the keys and their end
@pytest.mark.parametrize("end", ["low", "high"])
@pytest.mark.parametrize("far", ["none", "one", "both"])  # the other end's key: on no, one side
def test_unsampled_key_of_the_other_end(judge, exact, gap, end, far):
    n = 100_000
    g = torch.Generator().manual_seed(9)
    kr = torch.randperm(n, generator=g)
    ks = torch.randint(0, n, (2 * n,), generator=g)
    base = INFO.min + gap if end == "low" else INFO.max - gap - (n - 1)
    kr, ks = kr + base, ks + base
    if exact:
        # unsampled rows of one batch, more than its sampled region has room for
        rows = torch.arange(2 * n)
        ks[(rows % STRIDE != OFF_S) & (rows < n)] = base + n // 2
    other = INFO.max if end == "low" else INFO.min
    at_r, at_s = OFF + 1 + 20 * STRIDE, OFF_S + 1 + (n // 10 + 30) * STRIDE
    if far != "none":
        ks[at_s] = other
    if far == "both":
        kr[at_r] = other
    ir, is_ = torch.arange(n), torch.arange(2 * n)
    got = api.join_inner(*(t.to(DEV) for t in (kr, ir, ks, is_)), mem_budget_bytes=4 << 20,
                         router="pla", partitions=64, sample_stride=STRIDE, seed=SEED,
                         radix_judge=judge)
    if exact:
        assert api.stats()["route_regions"] == 3
    assert_pairs_equal(got, oracle.join_inner(kr.numpy(), ir.numpy(), ks.numpy(), is_.numpy()))
