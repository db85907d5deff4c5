"""GPU parity of batched joins over folded rows: pairs of one key value, of key
ranges that take one to three passes, 64-bit keys beside 32-bit ids, and ids that
fit no word (the batch then runs on columns), among empty and disjoint pairs."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_21237_gb300 import api
from gpu_util import DEV, assert_pairs_equal, np_of

pytestmark = pytest.mark.gpu

SIZES = [(3072, 6144), (60_000, 3072), (1, 30_000), (0, 5_000), (30_000, 0), (6_144, 100_001),
         (50_000, 50_000), (9_000, 2_900)]


@pytest.mark.parametrize("dtype,bits", [(torch.int32, 31), (torch.int32, 16), (torch.int64, 21),
                                        (torch.int64, 46), (torch.int64, 63)])
@pytest.mark.parametrize("ids", ["positions", "one_far"])
def test_batch_words(dtype, bits, ids):
    g = torch.Generator().manual_seed(bits)
    info = torch.iinfo(dtype)
    r_off, s_off, kr, ks, ir, is_ = [0], [0], [], [], [], []
    for j, (a, b) in enumerate(SIZES):
        # values of j's own range: one value, a few bits, ..., all of them; the last pair disjoint
        nb = min(bits, [3, 9, 0, 5, 5, 12, bits, 10][j])
        vals = torch.randint(0, min(1 << nb, (1 << 63) - 1), (max(a, 1),), generator=g, dtype=torch.int64)
        low = -(1 << (nb - 1)) if nb else 7
        kr.append((vals[:a] + low).to(dtype))
        pick = vals[torch.randint(0, max(a, 1), (b,), generator=g)]
        other = torch.randint(0, min(1 << nb, (1 << 63) - 1), (b,), generator=g, dtype=torch.int64)
        k = torch.where(torch.rand(b, generator=g) < (0.02 if nb < 12 else 0.5), pick, other) + low
        ks.append((k + (1 << 12) if j == 7 else k).to(dtype))
        ir.append(torch.arange(a, dtype=dtype))
        is_.append(torch.arange(b, dtype=dtype))
        r_off.append(r_off[-1] + a)
        s_off.append(s_off[-1] + b)
    kr, ks, ir, is_ = (torch.cat(x) for x in (kr, ks, ir, is_))
    if ids == "one_far":  # no row that the statistics sample
        is_[s_off[6] + 4321] = info.max
        ir[r_off[6] + 1234] = info.min
    pairs, off = api.join_batch(r_off, s_off, *(t.to(DEV) for t in (kr, ir, ks, is_)))
    exp, eoff = oracle.join_batch(np.array(r_off), np.array(s_off), kr.numpy(), ir.numpy(),
                                  ks.numpy(), is_.numpy())
    assert np.array_equal(np_of(off), eoff)
    assert_pairs_equal(pairs, exp)
