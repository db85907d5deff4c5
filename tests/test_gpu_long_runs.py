"""GPU parity of joins whose R has long runs of equal keys in chunks that are searched:
runs of every length around the doubling steps, runs that end with a chunk or go on in
the next; and the time
that meeting them takes."""
import pytest
import torch

import oracle
from paper_2602_21237_gb300 import api, datagen
from gpu_util import DEV, assert_pairs_equal

pytestmark = pytest.mark.gpu

LAYOUTS = [(torch.int32, "near"), (torch.int64, "near"), (torch.int64, "wide"),
           (torch.int64, "far")]


def columns(kr, ks, dtype, ids, gap):
    if ids == "wide":  # values spread over 64 bits: a key beside a 32-bit id
        kr, ks = datagen.scatter64(kr), datagen.scatter64(ks)
    else:
        kr, ks = kr * gap, ks * gap
    ir, is_ = torch.arange(kr.numel()), torch.arange(ks.numel())
    if ids == "far":
        ir, is_ = ir * (1 << 40), is_ * (1 << 40)
    return [t.to(dtype) for t in (kr, ir, ks, is_)]


@pytest.mark.parametrize("dtype,ids", LAYOUTS)
@pytest.mark.parametrize("ns", [40, 20_000])  # short S tiles, whole ones
def test_runs_of_every_length(dtype, ids, ns):
    g = torch.Generator().manual_seed(ns)
    lengths = [1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 31, 33, 63, 64, 65, 127, 129, 511, 513,
               1023, 1024, 1025, 2047, 2048, 2049, 2303, 2304, 4095, 4097, 4607, 4609, 6145, 8193]
    kr = torch.cat([torch.full((n,), 2 * i, dtype=torch.int64) for i, n in enumerate(lengths)])
    kr = kr[torch.randperm(kr.numel(), generator=g)]
    # every value and the gaps between a few times, the rest past all of them
    ks = torch.cat([torch.arange(-1, 2 * len(lengths) + 1),
                    2 * len(lengths) + torch.randint(1, 50_000, (ns,), generator=g)])
    ks = ks[torch.randperm(ks.numel(), generator=g)]
    cols = columns(kr, ks, dtype, ids, 40_000)
    got = api.join_inner(*(c.to(DEV) for c in cols), router="single")
    assert_pairs_equal(got, oracle.join_inner(*(c.numpy() for c in cols)))


@pytest.mark.parametrize("dtype", [torch.int32, torch.int64])
def test_time_does_not_grow_with_the_runs(dtype):
    # the same join with and without its matches (0.1% of S meets runs of about 2000 R
    # rows): a run's end takes a few steps more, not a walk of the run
    n_r, n_s, values = 10_000_000, 1_000_000, 5_000
    g = torch.Generator(device=DEV).manual_seed(3)
    kr = torch.randint(0, values, (n_r,), generator=g, device=DEV)
    ks = torch.randint(0, 1000 * values, (n_s,), generator=g, device=DEV)
    out = torch.empty((2 * n_r, 2), dtype=dtype, device=DEV)
    ir, is_ = (torch.arange(n, device=DEV, dtype=dtype) for n in (n_r, n_s))

    def best(k_r, k_s):
        t = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            api.join_inner(k_r.to(dtype), ir, k_s.to(dtype), is_, out=out)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        return min(t)

    none = best(kr * 1000, ks + (ks % 1000 == 0).to(ks.dtype))
    some = best(kr * 1000, ks)
    assert some < 1.4 * none, (some, none)
