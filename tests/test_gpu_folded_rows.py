"""GPU parity of the passes over folded rows (a row as one 64-bit word): tile
edges of both tile sizes, ids and keys that just fit a word or just do not (the
call then runs on separate columns), every consumer of folded rows."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_21237_gb300 import api, datagen
from gpu_util import DEV, assert_pairs_equal, np_of

pytestmark = pytest.mark.gpu

SMALL, LARGE = 4096, 8192  # rows of the two word tiles


def sorted_as_oracle(keys, ids):
    k, i = keys.to(DEV), ids.to(DEV)
    api.sort(k, i)
    ek, ei = oracle.sort(keys.numpy(), ids.numpy())
    assert np.array_equal(np_of(k), ek) and np.array_equal(np_of(i), ei)


@pytest.mark.parametrize("n", [SMALL - 1, SMALL, SMALL + 1, 5 * SMALL + 7, (1 << 22) - 1,
                               513 * LARGE, 513 * LARGE + 1])
@pytest.mark.parametrize("bits", [3, 27, 33, 64])
def test_tile_edges(n, bits):
    # at 2^22 rows the large tile and the plan of fewest pass units take over;
    # 33 key bits leave the key in both halves of the word, 64 do not fold: the
    # key travels beside a 32-bit id
    g = torch.Generator().manual_seed(n + bits)
    keys = torch.randint(-(1 << (bits - 1)), (1 << (bits - 1)) - 1, (n,), generator=g)
    sorted_as_oracle(keys, torch.arange(n))


@pytest.mark.parametrize("dtype", [torch.int32, torch.int64])
@pytest.mark.parametrize("ids", ["full", "one_far", "offset", "negative"])
@pytest.mark.parametrize("bits", [40, 63])
def test_ids_that_fit_and_that_do_not(dtype, ids, bits):
    # 40 key bits leave 24 id bits: positions of 2^17 rows fit, wherever they
    # start; one id far from the sampled ones does not, nor do full-range ids.
    # 63 key bits leave the key beside a 32-bit id, or a full one.
    n = 1 << 17
    info = torch.iinfo(dtype)
    g = torch.Generator().manual_seed(4)
    top = bits if dtype == torch.int64 else 30
    keys = torch.randint(0, (1 << top) - 1, (n,), generator=g, dtype=torch.int64).to(dtype)
    v = torch.arange(n, dtype=torch.int64)
    if ids == "full":
        v = torch.randint(info.min, info.max, (n,), generator=g, dtype=torch.int64)
    elif ids == "one_far":
        v[n // 2 + 17] = info.max
    elif ids == "offset":
        v = v + (info.max - n)
    else:
        v = -v * 3
    sorted_as_oracle(keys, v.to(dtype))
    kr, ks = keys[: n // 4], keys[torch.randint(0, n // 4, (n,), generator=g)]
    ir, is_ = v[n // 4: n // 2].to(dtype), v.to(dtype)
    exp = oracle.join_inner(kr.numpy(), ir.numpy(), ks.numpy(), is_.numpy())
    for router in ("single", "radix", "pla"):
        got = api.join_inner(kr.to(DEV), ir.to(DEV), ks.to(DEV), is_.to(DEV), router=router)
        assert_pairs_equal(got, exp)


@pytest.mark.parametrize("far", [0, 1 << 20, 1 << 45])
def test_keys_outside_the_sampled_window(far):
    # a budget below one sorted copy: the range is read off the sample; keys
    # past its slack send the join back to separate columns
    n, stride, seed = 200_000, 10, 5
    off = (((seed * 0x9E3779B97F4A7C15) % (1 << 64)) >> 33) % stride
    g = torch.Generator().manual_seed(9)
    kr = torch.randperm(n, generator=g)
    ks = torch.randint(0, n, (2 * n,), generator=g)
    kr[off + 1] = n + far
    ks[off + 2] = n + far
    kr[off + 3] = -far
    ir, is_ = torch.arange(n), torch.arange(2 * n)
    got = api.join_inner(*(t.to(DEV) for t in (kr, ir, ks, is_)), mem_budget_bytes=6 << 20,
                         router="pla", partitions=64, sample_stride=stride, seed=seed)
    assert api.stats()["scratch_peak"] <= 6 << 20
    assert_pairs_equal(got, oracle.join_inner(kr.numpy(), ir.numpy(), ks.numpy(), is_.numpy()))


@pytest.mark.parametrize("parts", [64, 1024])
def test_cut_table_route_and_lsd_batches(parts):
    # log-normal keys under learned cuts: batches of every width, most of them
    # sorted by LSD word passes; many-to-many
    kr, ir = datagen.lognormal_mix(1 << 17, 91, key_bits=34)
    ks, is_ = datagen.lognormal_mix((1 << 18) + 5, 92, key_bits=34)
    got = api.join_inner(*(t.to(DEV) for t in (kr, ir, ks, is_)), router="pla", partitions=parts,
                         radix_judge=-1)
    assert_pairs_equal(got, oracle.join_inner(kr.numpy(), ir.numpy(), ks.numpy(), is_.numpy()))
