"""GPU parity of gathers from columns that L2 holds, holds in part and cannot hold, with
few pairs (one launch) and many (large columns apart), against plain indexing; an id
out of range is reported whichever launch meets it.  The columns are made on the GPU."""
import pytest
import torch

from paper_2602_21237_gb300 import api
from gpu_util import DEV

pytestmark = pytest.mark.gpu

N_R, N_S = 70_000_000, 30_000_001  # 8-byte columns of 560 and 240 MB


@pytest.fixture(scope="module")
def columns():
    g = torch.Generator(device=DEV).manual_seed(7)
    wide = torch.randint(-(1 << 62), 1 << 62, (N_R,), generator=g, device=DEV)
    rc = [wide, wide.view(torch.float64), torch.arange(N_R, device=DEV, dtype=torch.int32)]
    sc = [torch.randint(-(1 << 62), 1 << 62, (N_S,), generator=g, device=DEV),
          torch.rand(N_S, generator=g, device=DEV, dtype=torch.float32),
          torch.arange(N_S, device=DEV)]
    return rc, sc


@pytest.mark.parametrize("n", [1, 1023, 100_003, (1 << 20) - 1, 1 << 20, 1_900_000, 5_000_001])
@pytest.mark.parametrize("dtype", [torch.int32, torch.int64])
def test_large_columns(columns, n, dtype):
    rc, sc = columns
    g = torch.Generator(device=DEV).manual_seed(n)
    pairs = torch.stack([torch.randint(0, m, (n,), generator=g, device=DEV)
                         for m in (N_R, N_S)], 1).to(dtype).contiguous()
    rows = pairs.to(torch.int64)
    for r, s in ((rc, sc), (rc[2:], sc[1:2]), (rc[:1], []), ([], sc)):
        got_r, got_s = api.gather_pairs(pairs, r, s, n_r=N_R, n_s=N_S)
        for side, (got, cols) in enumerate(((got_r, r), (got_s, s))):
            for x, c in zip(got, cols):
                # (bytes: a column of any bit patterns as floats holds NaNs)
                assert torch.equal(x.view(torch.uint8), c[rows[:, side]].view(torch.uint8))


@pytest.mark.parametrize("n", [1000, 5_000_001])
@pytest.mark.parametrize("side", [0, 1])
def test_id_out_of_range(columns, n, side):
    rc, sc = columns
    pairs = torch.zeros((n, 2), dtype=torch.int64, device=DEV)
    pairs[n // 2, side] = N_S if side else N_R
    with pytest.raises(api.TjError, match="out of range"):
        api.gather_pairs(pairs, rc, sc)
