"""The tensor-core path's rotation and its product of several matrices at once, at ragged batches and uneven row tiles."""
import numpy as np
import pytest
import torch

import oracle
import paper_2411_17525_b200 as hb
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,K", [(17, 1024), (40, 3072), (257, 2048), (300, 1024)])     # padding tokens, two token tiles
def test_blocked_rotation_equals_the_plain_transform(B, K):
    d = hb.make_desc(2, 256, 128, K, 4321)
    x = torch.randn(B, K, device="cuda", generator=torch.Generator(device="cuda").manual_seed(B)).to(torch.bfloat16)
    BN = hb.higgs_rotated_layout(d, B)
    got = hb.higgs_rotate_activations(d, x).view(-1, K // 64, BN // 8, 8, 8, 8)          # [tile][step][block][core][token][input]
    got = got.permute(0, 2, 4, 1, 3, 5).reshape(-1, K)
    assert torch.equal(got[:B], hb.higgs_rht(d, x, normalised=True).to(torch.float16))
    assert not got[B:].any()


@pytest.mark.parametrize("p,n,Ns,K,B,dtype", [
    (2, 256, (1024, 128, 128), 4096, 64, torch.float32),      # K split over clusters of eight
    (2, 64, (4096, 1024, 1024), 4096, 16, torch.bfloat16),    # from nine tokens when the concatenation is large enough
    (2, 16, (128, 2048), 1024, 257, torch.float32),           # two token tiles
    (1, 16, (256, 384, 128, 512), 2048, 33, torch.float32),   # four matrices
    (1, 256, (9600, 9600), 1024, 40, torch.bfloat16),         # no K split, more tiles than SMs
])
def test_matrices_of_one_tensor_core_launch(p, n, Ns, K, B, dtype):
    rng = np.random.default_rng(K + B)
    g64, gt = U.grid32(p, n)
    x = torch.from_numpy(rng.standard_normal((B, K)).astype(np.float32)).to(U.dev()).to(torch.bfloat16)
    descs, packed, scales, codes, sc16 = [], [], [], [], []
    for N in Ns:
        c = rng.integers(0, n, size=(N, K // p))
        s = (0.5 + rng.random((N, K // 1024))).astype(np.float16)
        d = hb.make_desc(p, n, N, K, 11)
        descs.append(d); codes.append(c); sc16.append(s)
        packed.append(hb.higgs_pack_codes(d, torch.from_numpy(c.astype(np.uint8)).to(U.dev())))
        scales.append(hb.scales_to_tile_major(torch.from_numpy(s).to(U.dev())))
    ys = [torch.full((B, N), float("nan"), dtype=dtype, device=U.dev()) for N in Ns]
    m = hb.MultiLinear(descs, packed, scales, gt, ys, B)
    hb.higgs_linear_multi(m, x)
    assert hb.higgs_device_status() == hb.HIGGS_OK
    assert m.launches == 2
    tol = 2e-3 + (2.0 ** -8 if dtype == torch.bfloat16 else 0.0)
    for d, y, pk, sc, c, s in zip(descs, ys, packed, scales, codes, sc16):
        alone = hb.higgs_linear(d, x, pk, sc, gt, out_dtype=dtype)
        assert U.linear_error(y.float().cpu().numpy(), alone.float().cpu().numpy().astype(np.float64)) <= tol
        rows = np.unique(np.r_[0, 15, 127, d.N - 128, d.N - 1, rng.integers(0, d.N, 6)])
        ref = oracle.linear_dense(x.float().cpu().numpy().astype(np.float64), c[rows].astype(np.int32), s[rows].astype(np.float64), 1024, g64, 11)
        assert U.linear_error(y[:, torch.from_numpy(rows).to(U.dev())].float().cpu().numpy(), ref) <= tol
