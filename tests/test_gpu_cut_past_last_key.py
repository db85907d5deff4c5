"""GPU parity of joins routed by a cut table whose last cut lies after the largest key (it
repeats among the sample's quantiles and gets a batch of its own) when the keys' range is a
power of two: no key that folds reaches that cut, the padding rows of a tile neither."""
import pytest
import torch

import oracle
from paper_2602_21237_gb300 import api
from gpu_util import DEV, assert_pairs_equal

pytestmark = pytest.mark.gpu

MIN, MAX = -(1 << 63), (1 << 63) - 1


@pytest.mark.parametrize("bits", [1, 2, 3, 8, 11, 17])
@pytest.mark.parametrize("n_r,n_s", [(28, 1), (754, 21), (4258, 231), (8192, 8192), (8193, 4_001),
                                     (180_000, 2)])
@pytest.mark.parametrize("base", [0, -171, MIN, "max"])
@pytest.mark.parametrize("budget", [0, 2 << 20])
def test_last_cut(bits, n_r, n_s, base, budget):
    g = torch.Generator().manual_seed(bits + n_r)
    base = MAX - (1 << bits) + 1 if base == "max" else base
    top = (1 << bits) - 1
    # every value once where there is room, the largest one often on R's side
    kr = torch.cat([torch.arange(top + 1), torch.full((n_r,), top)])[-n_r:] if n_r > top else \
        torch.full((n_r,), top)
    if n_r > 2 * (top + 1):
        kr[: n_r // 2] = torch.arange(n_r // 2) % (top + 1)
    kr = kr[torch.randperm(n_r, generator=g)]
    ks = torch.randint(0, top + 1, (n_s,), generator=g)
    ks[0] = 0 if n_s > 1 else top
    if n_s * n_r > 5_000_000:  # few pairs of the heavy key
        ks = torch.where(ks == top, torch.zeros_like(ks), ks)
        ks[:1] = top
    kr, ks = kr + base, ks + base
    ir, is_ = torch.arange(n_r), torch.arange(n_s)
    exp = oracle.join_inner(kr.numpy(), ir.numpy(), ks.numpy(), is_.numpy())
    for stride in (1, 100):
        got = api.join_inner(*(t.to(DEV) for t in (kr, ir, ks, is_)), router="pla",
                             mem_budget_bytes=budget, sample_stride=stride, radix_judge=-1.0)
        assert_pairs_equal(got, exp)
