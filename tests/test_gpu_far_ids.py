"""Joins and sorts of 64-bit rows of which some ids lie outside the range that a sample
gives (sentinels): parity for ids at the edges of the window of foldable ids, for as many
as the table of far ids holds and one more, in every operation; and the time of such calls
against ids that never fold."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_21237_gb300 import api
from gpu_util import DEV, assert_pairs_equal, np_of

pytestmark = pytest.mark.gpu

FAR, ROOM = -(1 << 62), 2048
TILE = 3072                  # rows of a tile, of which the sample takes the first and last
LARGE = (1 << 22) + 4097     # many tiles a CTA, large word tiles
SMALL = 70_000


def unsampled(n, count, seed):
    g = torch.Generator().manual_seed(seed)
    rows = torch.randperm(n, generator=g)
    if n > 1216 * TILE:
        rows = rows[(rows % TILE > 0) & (rows % TILE < TILE - 1)]
    return rows[:count]


def sort_check(keys, ids):
    k, i = keys.to(DEV), ids.to(DEV)
    api.sort(k, i)
    ek, ei = oracle.sort(keys.numpy(), ids.numpy())
    assert np.array_equal(np_of(k), ek) and np.array_equal(np_of(i), ei)


@pytest.mark.parametrize("n", [SMALL, LARGE])
@pytest.mark.parametrize("count", [1, 300, ROOM, ROOM + 1, 9000])
@pytest.mark.parametrize("bits", [23, 50, 63])  # folded, wide (prefix sort), wide
def test_sort(n, count, bits):
    g = torch.Generator().manual_seed(bits)
    keys = torch.randint(0, (1 << bits) - 1, (n,), generator=g)
    ids = torch.arange(n)
    at = unsampled(n, count, count + bits)
    ids[at] = FAR + torch.arange(at.numel()) // 3
    sort_check(keys, ids)


@pytest.mark.parametrize("n", [SMALL, LARGE])
@pytest.mark.parametrize("bits", [23, 30, 63])
def test_edges_of_the_window(n, bits):
    # offsets: [0, esc) ids, [esc, top] codes of far ids, as which such ids are far too
    g = torch.Generator().manual_seed(n + bits)
    keys = torch.randint(0, (1 << bits) - 1, (n,), generator=g)
    keys[0], keys[1] = 0, (1 << bits) - 1
    avail = 64 - bits if bits < 40 else 32
    top = (1 << avail) - 1
    esc = 1 << (avail - 1)
    ilo = -((esc - 1 - (n - 1)) // 2)
    edges = [ilo - 1, ilo, ilo + 1, ilo + esc - 1, ilo + esc, ilo + esc + 1, ilo + esc + 7, ilo + esc + ROOM,
             ilo + top, ilo + top + 1, FAR, -FAR]
    at = unsampled(n, 5 * len(edges), 3)
    ids = torch.arange(n)
    ids[at] = torch.tensor(edges).repeat(5)
    ids[0], ids[n - 1] = 0, n - 1
    sort_check(keys, ids)


def join_columns(n_r, n_s, count, seed):
    g = torch.Generator().manual_seed(seed)
    kr = torch.randperm(n_r, generator=g)
    kr[: n_r // 10] = kr[n_r // 10: 2 * (n_r // 10)]  # some keys twice
    ks = torch.randint(0, n_r, (n_s,), generator=g)
    ids = [torch.arange(n_r), torch.arange(n_s)]
    for side, n in enumerate((n_r, n_s)):
        at = unsampled(n, count, seed + side)
        ids[side][at] = FAR + 5 * torch.arange(at.numel()) + side
    return kr, ids[0], ks, ids[1]


@pytest.mark.parametrize("n_r,n_s", [(9_000, 20_001), (1_000_003, 3_500_001)])
@pytest.mark.parametrize("count", [1, ROOM // 2, ROOM])
@pytest.mark.parametrize("router,budget", [("single", 0), ("radix", 0), ("pla", 0), ("pla", 1)])
@pytest.mark.parametrize("spread", [1, 1 << 18])  # folded rows, wide ones (one pass only)
def test_join(n_r, n_s, count, router, budget, spread):
    kr, ir, ks, is_ = join_columns(n_r, n_s, count, 11)
    got = api.join_inner(*(t.to(DEV) for t in (kr * spread, ir, ks * spread, is_)),
                         mem_budget_bytes=12 * (n_r + n_s) + (1 << 20) if budget else 0,
                         router=router)
    assert_pairs_equal(got, oracle.join_inner(kr.numpy(), ir.numpy(), ks.numpy(), is_.numpy()))


@pytest.mark.parametrize("count", [1, 100, ROOM])
@pytest.mark.parametrize("spread", [1, 1 << 40])
def test_batch(count, spread):
    jobs = [join_columns(n_r, n_s, count, 20 + n_r) for n_r, n_s in ((7_000, 30_000), (20_000, 9_000))]
    kr, ir, ks, is_ = (torch.cat([j[c] for j in jobs]) for c in range(4))
    kr, ks = kr * spread, ks * spread
    r_off, s_off = np.array([0, 7_000, 27_000]), np.array([0, 30_000, 39_000])
    pairs, off = api.join_batch(r_off.tolist(), s_off.tolist(),
                                *(t.to(DEV) for t in (kr, ir, ks, is_)))
    exp, eoff = oracle.join_batch(r_off, s_off, kr.numpy(), ir.numpy(), ks.numpy(), is_.numpy())
    assert np.array_equal(np_of(off), eoff)
    assert_pairs_equal(pairs, exp)


def best(call, reps=20):
    t = []
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        call()
        b.record()
        b.synchronize()
        t.append(a.elapsed_time(b))
    return min(t)


@pytest.mark.parametrize("n", [30_000, 1_000_000, 30_000_000])
@pytest.mark.parametrize("op", ["sort", "join"])
def test_one_far_id_costs_no_second_run(n, op):
    # ids of any value take separate columns at once; a far id among others must not
    # cost a folding pass and a wait before the same
    g = torch.Generator(device=DEV).manual_seed(n)
    keys = torch.randperm(n, generator=g, device=DEV)
    one = torch.arange(n, device=DEV)
    one[n // 2 + 345] = FAR
    any_ = torch.randint(FAR, -FAR, (n,), generator=g, device=DEV)
    kr, ir = keys[: n // 3].clone(), torch.arange(n // 3, device=DEV)
    out = torch.empty((n, 2), dtype=torch.int64, device=DEV)
    call = (lambda ids: api.sort(keys.clone(), ids.clone())) if op == "sort" else \
        (lambda ids: api.join_inner(kr, ir, keys, ids, out=out))
    t_any, t_one = best(lambda: call(any_)), best(lambda: call(one))
    assert t_one < 1.2 * t_any, (t_one, t_any)
