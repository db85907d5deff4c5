"""GPU parity of joins under learned cuts whose keys span (nearly) all of int64: the uniform
index over the cuts has its last bucket at the end of the 64-bit offsets, where most of the
keys and cuts lie here."""
import pytest
import torch

import oracle
from paper_2602_21237_gb300 import api
from gpu_util import DEV, assert_pairs_equal

pytestmark = pytest.mark.gpu

MIN, MAX = -(1 << 63), (1 << 63) - 1


@pytest.mark.parametrize("top", [1 << 20, 1 << 45, 1 << 52, 1 << 56, 1 << 62])
@pytest.mark.parametrize("gap", [0, 1, 1 << 52, 1 << 54])  # between the keys and either end
@pytest.mark.parametrize("router,budget", [("pla", 0), ("pla", 4 << 20), ("mlp", 0)])
def test_keys_in_the_last_bucket(top, gap, router, budget):
    n_r, n_s = 60_000, 250_000
    g = torch.Generator().manual_seed(top % 1009)
    kr = MAX - gap - torch.randint(0, top, (n_r,), generator=g)
    kr[::50] = torch.randint(-(1 << 62), 1 << 62, (n_r // 50,), generator=g)
    kr[7], kr[11] = MIN + gap, MAX - gap
    ks = kr[torch.randint(0, n_r, (n_s,), generator=g)]
    ks[::3] = MAX - gap - torch.randint(0, top, (len(ks[::3]),), generator=g)
    ir, is_ = torch.arange(n_r), torch.arange(n_s)
    got = api.join_inner(*(t.to(DEV) for t in (kr, ir, ks, is_)), router=router,
                         mem_budget_bytes=budget, radix_judge=-1.0)
    assert_pairs_equal(got, oracle.join_inner(kr.numpy(), ir.numpy(), ks.numpy(), is_.numpy()))
