"""GPU parity of the resident join on separate columns (64-bit ids of any value do not
fold): S rows of a sub-batch at the edges of a thread's two groups of rows, of a warp's
rows and of a tile; one and several R rows a key."""
import pytest
import torch

import oracle
from paper_2602_21237_gb300 import api
from gpu_util import DEV, assert_pairs_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns", [1, 33, 287, 288, 289, 575, 576, 577, 2304, 2593, 4607, 4608, 4609,
                                9217])
@pytest.mark.parametrize("copies", [1, 2])
def test_rows_of_a_sub_batch(ns, copies):
    g = torch.Generator().manual_seed(ns)
    # two batches of 1024 keys, each one sub-batch
    kr = torch.randperm(2048, generator=g)[:900].repeat(copies)
    ks = torch.cat([torch.randint(0, 1024, (ns,), generator=g),
                    torch.randint(1024, 2048, (500,), generator=g),
                    torch.tensor([0, 2047])])
    ks = ks[torch.randperm(ks.numel(), generator=g)]
    ir, is_ = (torch.randint(-(1 << 62), 1 << 62, k.shape, generator=g) for k in (kr, ks))
    got = api.join_inner(*(t.to(DEV) for t in (kr, ir, ks, is_)), router="radix", partitions=2)
    assert api.stats()["fused_batches"] == 2
    assert_pairs_equal(got, oracle.join_inner(kr.numpy(), ir.numpy(), ks.numpy(), is_.numpy()))
