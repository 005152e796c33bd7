"""Dequantisation and layer error straight from the packed stream, at the sizes where the kernel's work split and lane
mapping can go wrong: one tile, groups that are no multiple of the stride, one more turn than there are blocks."""
import numpy as np
import pytest
import torch

import oracle
import paper_2411_17525_b200 as hb
from tests import gpu_util as U

pytestmark = pytest.mark.gpu
G = 1024
GRIDS = [(2, 256), (2, 64), (2, 16), (1, 16), (1, 8), (1, 4), (1, 256)]


@pytest.mark.parametrize("p,n", GRIDS)
@pytest.mark.parametrize("N,K", [(16, 1024), (48, 3072), (1488, 7168)])      # 1, 9 and 651 turns
def test_packed_rows_match_oracle(p, n, N, K):
    rng = np.random.default_rng(N + n)
    codes = rng.integers(0, n, size=(N, K // p))
    sc16 = (0.5 + rng.random((N, K // G))).astype(np.float16)
    g64, gt = U.grid32(p, n)
    xi = 99 + n
    d = hb.make_desc(p, n, N, K, xi)
    packed = hb.higgs_pack_codes(d, torch.from_numpy(codes.astype(np.uint8)).to(U.dev()))
    scales = hb.scales_to_tile_major(torch.from_numpy(sc16).to(U.dev()))
    ref = oracle.dequantize(codes.astype(np.int32), sc16.astype(np.float64), G, g64, xi)
    got = hb.higgs_dequantize(d, packed, scales, gt).cpu().numpy().astype(np.float64)
    # fp32 butterflies: ten stages of one rounding each on values of the group's size
    assert np.max(np.abs(got - ref)) <= 10 * 2.0 ** -24 * 8 * np.sqrt(np.mean(ref ** 2))
    W = (ref + 0.1 * rng.standard_normal((N, K))).astype(np.float32)
    for dtype in (torch.float32, torch.bfloat16):
        Wt = torch.from_numpy(W).to(U.dev()).to(dtype)
        t2 = hb.higgs_layer_error(d, Wt, packed, scales, gt)
        t2_ref = oracle.layer_error(Wt.float().cpu().numpy().astype(np.float64), codes.astype(np.int32), sc16.astype(np.float64), G, g64, xi)
        assert abs(t2 - t2_ref) <= 1e-5 * t2_ref
        assert t2 == hb.higgs_layer_error(d, Wt, packed, scales, gt)          # partial sums are added in a fixed order
