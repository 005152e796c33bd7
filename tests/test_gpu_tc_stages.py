"""The tensor-core product at every code format and at token tiles that change the depth of its rings."""
import numpy as np
import pytest
import torch

import oracle
import paper_2411_17525_b200 as hb
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,n", [(2, 256), (2, 64), (1, 16), (2, 16), (1, 256)])
@pytest.mark.parametrize("N,K,B", [(128, 1024, 17), (256, 3072, 33), (128, 5120, 65), (128, 2048, 144), (384, 1024, 256), (19072, 1024, 257)])
def test_tensor_core_rings(p, n, N, K, B):
    """Rings shorter and longer than the layer, K split over a cluster or not, one or two token tiles."""
    rng = np.random.default_rng(n + B)
    g64, gt = U.grid32(p, n)
    c = rng.integers(0, n, size=(N, K // p))
    s = (0.5 + rng.random((N, K // 1024))).astype(np.float16)
    x = torch.from_numpy(rng.standard_normal((B, K)).astype(np.float32)).to(U.dev()).to(torch.bfloat16)
    d = hb.make_desc(p, n, N, K, 29)
    assert hb.higgs_rotated_layout(d, B) > 0
    packed = hb.higgs_pack_codes(d, torch.from_numpy(c.astype(np.uint8)).to(U.dev()))
    y = hb.higgs_linear(d, x, packed, hb.scales_to_tile_major(torch.from_numpy(s).to(U.dev())), gt)
    assert hb.higgs_device_status() == hb.HIGGS_OK
    rows = np.unique(np.r_[0:16, 127, N - 128, N - 1, rng.integers(0, N, 24)])
    ref = oracle.linear_dense(x.float().cpu().numpy().astype(np.float64), c[rows].astype(np.int32), s[rows].astype(np.float64), 1024, g64, 29)
    # fp16 roundings of table entry, scaled weight and rotated activation: 3 x 2^-11 of the norm each at worst
    assert U.linear_error(y[:, torch.from_numpy(rows).to(U.dev())].float().cpu().numpy(), ref) <= 3 * 2.0 ** -11


@pytest.mark.parametrize("p,n", [(2, 256), (2, 64)])
@pytest.mark.parametrize("N,K,B", [(4096, 1024, 1500), (6144, 2048, 1000), (2304, 3072, 1111)])
def test_token_tiles_that_cross_the_layouts(p, n, N, K, B):
    """The product's token tiles begin and end inside the layout's: every token against the same layer in batches of one tile."""
    rng = np.random.default_rng(B)
    _, gt = U.grid32(p, n)
    d = hb.make_desc(p, n, N, K, 31)
    assert straddles(d, B)
    packed = hb.higgs_pack_codes(d, torch.from_numpy(rng.integers(0, n, size=(N, K // p)).astype(np.uint8)).to(U.dev()))
    sc = hb.scales_to_tile_major(torch.from_numpy((0.5 + rng.random((N, K // 1024))).astype(np.float16)).to(U.dev()))
    x = torch.from_numpy(rng.standard_normal((B, K)).astype(np.float32)).to(U.dev()).to(torch.bfloat16)
    y = hb.higgs_linear(d, x, packed, sc, gt)
    ref = torch.cat([hb.higgs_linear(d, x[b:b + 256].contiguous(), packed, sc, gt) for b in range(0, B, 256)])
    assert hb.higgs_device_status() == hb.HIGGS_OK
    # the same fp16 operands; fp32 sums of K products in another order when a part is cut into K slices
    assert (y - ref).abs().max() <= 2.0 ** -24 * K * ref.abs().max()


def straddles(d, B):
    """Whether some token tile of the product lies across two of the layout's."""
    tile, layout = hb.higgs_linear_token_tile(d, B), hb.higgs_rotated_layout(d, B)
    return any(b // layout != (min(b + tile, B) - 1) // layout for b in range(0, B, tile))


def layer(p, n, N, K, seed, rng):
    d = hb.make_desc(p, n, N, K, seed)
    packed = hb.higgs_pack_codes(d, torch.from_numpy(rng.integers(0, n, size=(N, K // p)).astype(np.uint8)).to(U.dev()))
    return d, packed, hb.scales_to_tile_major(torch.from_numpy((0.5 + rng.random((N, K // 1024))).astype(np.float16)).to(U.dev()))


@pytest.mark.parametrize("p,n,dtype", [(2, 16, torch.float32), (1, 256, torch.float32), (2, 256, torch.bfloat16), (1, 256, torch.bfloat16)])
def test_straddling_tiles_of_every_format(p, n, dtype):
    N, K, B = 4096, 1024, 1500
    rng = np.random.default_rng(n)
    _, gt = U.grid32(p, n)
    d, packed, sc = layer(p, n, N, K, 31, rng)
    assert straddles(d, B)
    x = torch.from_numpy(rng.standard_normal((B, K)).astype(np.float32)).to(U.dev()).to(torch.bfloat16)
    y = hb.higgs_linear(d, x, packed, sc, gt, out_dtype=dtype).float()
    ref = torch.cat([hb.higgs_linear(d, x[b:b + 256].contiguous(), packed, sc, gt) for b in range(0, B, 256)])
    assert hb.higgs_device_status() == hb.HIGGS_OK
    # the same fp16 operands; fp32 sums of K products in another order when a part is cut into K slices; one rounding to bf16
    assert ((y - ref).abs() <= 2.0 ** -24 * K * ref.abs().max() + (2.0 ** -8 * ref.abs() if dtype == torch.bfloat16 else 0.0)).all()


def test_straddling_tiles_of_several_matrices():
    Ns, K, B = (1024, 128, 2944), 1024, 1500
    rng = np.random.default_rng(5)
    _, gt = U.grid32(2, 256)
    assert straddles(hb.make_desc(2, 256, sum(Ns), K, 31), B)
    layers = [layer(2, 256, N, K, 31, rng) for N in Ns]
    x = torch.from_numpy(rng.standard_normal((B, K)).astype(np.float32)).to(U.dev()).to(torch.bfloat16)
    ys = [torch.full((B, N), float("nan"), device=U.dev()) for N in Ns]
    m = hb.MultiLinear([a[0] for a in layers], [a[1] for a in layers], [a[2] for a in layers], gt, ys, B)
    hb.higgs_linear_multi(m, x)
    assert hb.higgs_device_status() == hb.HIGGS_OK and m.launches == 2
    for (d, packed, sc), y in zip(layers, ys):
        ref = torch.cat([hb.higgs_linear(d, x[b:b + 256].contiguous(), packed, sc, gt) for b in range(0, B, 256)])
        assert (y - ref).abs().max() <= 2.0 ** -24 * K * ref.abs().max()


def test_straddling_tiles_into_a_wider_output():
    """A row shard's columns of two destinations; everything beside them stays as it was."""
    N, K, B, ld, at = 4096, 1024, 1500, 4096 + 640, 512
    rng = np.random.default_rng(6)
    _, gt = U.grid32(2, 64)
    d, packed, sc = layer(2, 64, N, K, 31, rng)
    assert straddles(d, B)
    x = torch.from_numpy(rng.standard_normal((B, K)).astype(np.float32)).to(U.dev()).to(torch.bfloat16)
    outs = [torch.full((B, ld), -7.0, device=U.dev()) for _ in range(2)]
    hb.higgs_linear_gather(d, x, packed, sc, gt, outs, at)
    assert hb.higgs_device_status() == hb.HIGGS_OK
    ref = hb.higgs_linear(d, x, packed, sc, gt)
    for o in outs:
        assert torch.equal(o[:, at:at + N], ref)
        assert (o[:, :at] == -7.0).all() and (o[:, at + N:] == -7.0).all()
