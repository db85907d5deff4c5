"""GPU parity of sorts by a key prefix (three digits of the leading bits, then the
runs of equal prefixes put in order): duplicates, runs at and over the longest one
that is put in order, at tile edges, in order and not, folded and wide rows."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_21237_gb300 import api, datagen
from gpu_util import DEV, np_of

pytestmark = pytest.mark.gpu

MAX, TILE = 256, 4096  # longest run put in order, rows of a tile
LARGE = (1 << 22) + 5000  # rows that a sample of 2048 sees few of a run's


def check(keys, passes):
    ids = torch.arange(keys.numel())
    k, i = keys.to(DEV), ids.to(DEV)
    api.sort(k, i)
    ek, ei = oracle.sort(keys.numpy(), ids.numpy())
    assert np.array_equal(np_of(k), ek) and np.array_equal(np_of(i), ei)
    got = api.stats()["radix_passes"]
    assert (got == 3) == passes, got


@pytest.mark.parametrize("n", [1 << 17, (1 << 17) + 4097, LARGE])
@pytest.mark.parametrize("bits", [45, 64])
def test_nearly_unique_keys(n, bits):
    # 2^17 rows of 45-bit keys fold, 64-bit keys travel beside 32-bit ids; every
    # 16th key comes twice
    g = torch.Generator().manual_seed(n)
    keys = datagen.scatter64(torch.randperm(n, generator=g))
    m = n // 16 * 16
    keys[:m:16] = keys[1:m:16]
    check(keys >> (64 - bits), True)


def test_few_distinct_keys_take_every_digit():
    g = torch.Generator().manual_seed(3)
    keys = datagen.scatter64(torch.randint(0, 1000, (1 << 17,), generator=g))
    check(keys, False)


@pytest.mark.parametrize("length", [2, MAX - 1, MAX, MAX + 1, MAX + 2, 2 * MAX + 100])
@pytest.mark.parametrize("kind", ["equal", "falling"])
@pytest.mark.parametrize("before", [0, 7 * TILE - 100, 7 * TILE])
def test_runs_at_tile_edges(length, kind, before):
    # `before` rows of smaller prefixes, then a run that shares one prefix: one
    # repeated key, or keys that fall in input order
    n = LARGE
    g = torch.Generator().manual_seed(length + before)
    step = (1 << 62) // n  # one prefix of 27 bits holds no two multiples of it
    other = torch.arange(n - length) * step
    run = torch.full((length,), (before * step) if before else 0)
    run += step // 2
    other[before:] += step
    if kind == "falling":
        run += torch.arange(length - 1, -1, -1)
    keys = torch.cat((other, run))
    pos = torch.randperm(n, generator=g)
    run_at = torch.sort(pos[n - length:]).values
    out = torch.empty(n, dtype=torch.int64)
    out[pos[: n - length]] = other
    out[run_at] = run
    check(out - (1 << 61), kind == "equal" or length <= MAX)
