"""GPU parity of tile joins whose S is sparse against R (short S tiles, searched on
chip): S sizes at the edges of the short tiles, runs of equal R keys that cross the
chunks of R, one pass and batched."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_21237_gb300 import api, datagen
from gpu_util import DEV, assert_pairs_equal, np_of

pytestmark = pytest.mark.gpu

SHAPES = [(200_000, 1), (200_000, 63), (200_000, 65), (200_000, 2_049), (300_000, 31_007),
          (300_001, 149_999), (300_000, 150_001), (9_000, 4_097)]


def columns(nr, ns, dtype, copies, ids):
    g = torch.Generator().manual_seed(nr + ns + copies)
    vals = torch.randint(0, max(2, 2 * nr // copies), (nr,), generator=g)
    ks = torch.randint(0, max(2, 2 * nr // copies), (ns,), generator=g)
    if dtype == torch.int64:  # values spread over 64 bits
        vals, ks = datagen.scatter64(vals), datagen.scatter64(ks)
    ir, is_ = torch.arange(nr), torch.arange(ns)
    if ids == "far":  # no 32-bit window holds them: separate columns
        ir, is_ = ir * (1 << 40), is_ * (1 << 40)
    return vals.to(dtype), ir.to(dtype), ks.to(dtype), is_.to(dtype)


@pytest.mark.parametrize("nr,ns", SHAPES)
@pytest.mark.parametrize("copies", [1, 60])
@pytest.mark.parametrize("dtype,ids", [(torch.int32, "near"), (torch.int64, "near"),
                                       (torch.int64, "far")])
def test_one_pass(nr, ns, copies, dtype, ids):
    cols = columns(nr, ns, dtype, copies, ids)
    exp = oracle.join_inner(*(c.numpy() for c in cols))
    got = api.join_inner(*(c.to(DEV) for c in cols), router="single")
    assert_pairs_equal(got, exp)


@pytest.mark.parametrize("copies", [1, 30])
@pytest.mark.parametrize("dtype", [torch.int32, torch.int64])
def test_batch(copies, dtype):
    jobs = [columns(nr, ns, dtype, copies, "near") for nr, ns in SHAPES]
    kr, ir, ks, is_ = (torch.cat([j[c] for j in jobs]) for c in range(4))
    r_off = np.concatenate([[0], np.cumsum([nr for nr, _ in SHAPES])])
    s_off = np.concatenate([[0], np.cumsum([ns for _, ns in SHAPES])])
    pairs, off = api.join_batch(r_off.tolist(), s_off.tolist(),
                                *(t.to(DEV) for t in (kr, ir, ks, is_)))
    exp, eoff = oracle.join_batch(r_off, s_off, kr.numpy(), ir.numpy(), ks.numpy(), is_.numpy())
    assert np.array_equal(np_of(off), eoff)
    assert_pairs_equal(pairs, exp)
