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
