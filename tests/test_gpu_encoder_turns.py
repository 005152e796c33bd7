"""The pruned encoder's split into turns against the exhaustive scan (which small calls take): an odd number of turns, one
more turn than there are half-blocks, groups that do not divide the stride, both input types, every output."""
import pytest
import torch

import paper_2411_17525_b200 as hb
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("p,n,N,K", [(2, 256, 2064, 1024), (1, 16, 688, 3072), (2, 64, 4816, 1024), (1, 256, 2128, 5120), (2, 16, 688, 7168)])
def test_turns_equal_the_exhaustive_scan(p, n, N, K, dtype):
    _, gt = U.grid32(p, n)
    W = torch.randn(N, K, device="cuda", generator=torch.Generator(device="cuda").manual_seed(N)).mul_(0.02)
    W[5, :1024] = 0.0                                    # a group of zeros
    W[7, 3] = 100.0                                      # one input carries the group: every rotated value at the table's edge
    W = W.to(dtype)
    d = hb.make_desc(p, n, N, K, 13)
    packed, scales, canon = hb.higgs_quantize(d, W, gt, want_canonical=True)
    alone, _, _ = hb.higgs_quantize(d, W, gt)
    assert torch.equal(packed, alone) and torch.equal(packed, hb.higgs_pack_codes(d, canon))
    step = 2032 // (K // 1024) // 16 * 16                # rows of a call that stays below the pruned search's threshold
    for r in range(0, N, step):
        rows = min(step, N - r)
        ds = hb.make_desc(p, n, rows, K, 13)
        _, sc, ca = hb.higgs_quantize(ds, W[r:r + rows].contiguous(), gt, want_canonical=True)
        assert torch.equal(canon[r:r + rows], ca) and torch.equal(scales[r // 16:(r + rows) // 16], sc)


@pytest.mark.parametrize("p,n", [(2, 256), (2, 16), (1, 16)])
def test_outermost_cells_of_the_search_table_are_never_used(p, n):
    """Points beyond the table fall into its outermost cells, so these are always scanned, whatever a table (an older one, say) lists there."""
    _, grid = U.grid32(p, n)
    W = torch.randn(2048, 4096, device=U.dev(), generator=torch.Generator(device="cuda").manual_seed(p))
    d = hb.make_desc(p, n, 2048, 4096, 3)
    table = hb.higgs_make_encoder_table(p, n, grid)
    cells = table.view(torch.int32).view(128, 128) if p == 2 else table.view(torch.int32).view(1, 1024)
    if p == 2:
        cells[[0, -1]] = 0
    cells[:, [0, -1]] = 0
    packed, scales, codes = hb.higgs_quantize(d, W, grid, want_canonical=True, table=table)
    few = hb.make_desc(p, n, 16, 4096, 3)                   # (small layers are scanned exhaustively)
    ref = torch.cat([hb.higgs_quantize(few, W[r:r + 16].contiguous(), grid, want_canonical=True)[2] for r in range(0, 2048, 16)])
    assert hb.higgs_device_status() == hb.HIGGS_OK
    assert torch.equal(codes, ref)
