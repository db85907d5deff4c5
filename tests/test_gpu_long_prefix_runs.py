"""GPU parity of sorts by a key prefix with long runs of equal prefixes out of order, which
are sorted by themselves: one and many, at both ends of the order, beside runs in order,
folded and wide rows, far ids among them; more than are listed (every digit, all rows)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_21237_gb300 import api, datagen
from gpu_util import DEV, np_of

pytestmark = pytest.mark.gpu

FAR = -(1 << 62)


def mixed(n, bits, lengths, kind, seed):
    """Hashed keys of `bits` bits, and runs of the given lengths that share a prefix each."""
    g = torch.Generator().manual_seed(seed)
    keys = datagen.scatter64(torch.randperm(n, generator=g)) >> (64 - bits)
    lo, hi = int(keys.min()), int(keys.max())
    rows = torch.randperm(n, generator=g)[: sum(lengths)]
    at = 0
    for r, length in enumerate(lengths):
        # runs spread over the range, the first and the last at its ends
        first = lo + (hi - lo - (1 << 17)) // max(1, len(lengths) - 1) * r
        if kind == "equal" or (kind == "some equal" and r % 2):
            run = torch.full((length,), first)
        else:
            run = first + torch.randint(0, 1 << 16, (length,), generator=g)
        keys[rows[at: at + length]] = run
        at += length
    return keys


def check(keys, ids=None):
    ids = torch.arange(keys.numel()) if ids is None else ids
    k, i = keys.to(DEV), ids.to(DEV)
    api.sort(k, i)
    ek, ei = oracle.sort(keys.numpy(), ids.numpy())
    assert np.array_equal(np_of(k), ek) and np.array_equal(np_of(i), ei)
    return api.stats()["radix_passes"]


@pytest.mark.parametrize("bits", [45, 64])  # 45 fold beside ids of up to 19 bits
@pytest.mark.parametrize("lengths", [[257], [900], [257, 300], [300, 257, 611, 258, 400, 1000]])
@pytest.mark.parametrize("kind", ["random", "some equal", "equal"])
def test_few_long_runs(bits, lengths, kind):
    n = 500_000 if bits == 45 else 3_000_000
    passes = check(mixed(n, bits, lengths, kind, len(lengths) + bits))
    # (a run of one key is in order, unless a hashed key shares its prefix)
    assert (3 if kind == "equal" else 4) <= passes <= 11


@pytest.mark.parametrize("n,rows", [(600_000, 4_000), (30_000_000, 2_000)])
def test_small_codes_among_hashed_keys(n, rows):
    g = torch.Generator(device=DEV).manual_seed(rows)
    keys = torch.randint(-(1 << 62), 1 << 62, (n,), generator=g, device=DEV)
    at = torch.randperm(n, generator=g, device=DEV)[:rows]
    keys[at] = torch.randint(0, 1000, (at.numel(),), generator=g, device=DEV)
    ids = torch.arange(n, device=DEV)
    k, i = keys.clone(), ids.clone()
    api.sort(k, i)
    ek, ei = torch.sort(keys, stable=True)
    assert torch.equal(k, ek) and torch.equal(i, ei)


def test_far_ids_in_long_runs():
    n = 3_000_000
    keys = mixed(n, 64, [300, 5000, 257], "random", 8)
    ids = torch.arange(n)
    g = torch.Generator().manual_seed(1)
    ids[torch.randperm(n, generator=g)[:50]] = FAR + torch.arange(50)
    run = torch.nonzero(keys < int(keys.min()) + (1 << 17)).flatten()
    ids[run[10:40]] = FAR - torch.arange(30)
    assert 3 < check(keys, ids) <= 11


def test_more_runs_than_are_listed():
    n = 14_000_000
    passes = check(mixed(n, 64, [260] * 1100, "random", 4))
    assert passes == 8
