"""The rotation kernel in front of the small-batch product."""
import pytest
import torch

import oracle
import paper_2411_17525_b200 as hb
from paper_2411_17525_b200 import binding
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,K", [(1, 1024), (2, 28672), (3, 3072), (8, 14336), (16, 2048)])
def test_rotation_in_fragment_order(B, K):
    xi, d = 977, hb.make_desc(2, 256, 16, K, 977)
    assert hb.higgs_rotated_layout(d, B) == 0
    x = torch.randn(B, K, device=U.dev(), generator=torch.Generator(device="cuda").manual_seed(K)).to(torch.bfloat16)
    x[0, :1024] *= 1e3
    # word t*8 + m*2 + h of a 64-input block is the pair 8m + 4h + t
    got = hb.higgs_rotate_activations(d, x).view(B, K // 64, 4, 4, 2, 2).permute(0, 1, 3, 4, 2, 5).reshape(B, K).double().cpu()
    sgn = torch.from_numpy(oracle.signs(xi, K)).double()
    H = torch.ones(1, 1, dtype=torch.float64)
    for _ in range(10):
        H = torch.cat([torch.cat([H, H], 1), torch.cat([H, -H], 1)], 0)
    xs = (x.double().cpu() * sgn).view(B, K // 1024, 1024)
    ref = (xs @ H / 32).reshape(B, K)
    # ten fp32 stages of one rounding each, below the sum of magnitudes, then one rounding to fp16
    bound = (10 * 2.0 ** -24 / 32 * xs.abs().sum(-1, keepdim=True)).expand(B, K // 1024, 1024).reshape(B, K)
    assert ((got - ref).abs() <= bound + 2.0 ** -11 * (ref.abs() + bound) + 2.0 ** -25).all()


@pytest.mark.parametrize("N,K,B,one_launch", [(16, 1024, 1, True), (512, 1024, 2, True), (512, 1024, 3, False), (256, 1024, 17, False)])
def test_a_call_without_workspace(N, K, B, one_launch):
    """One launch takes no workspace; everything else refuses to do without."""
    d = hb.make_desc(2, 256, N, K, 5)
    _, grid = U.grid32(2, 256)
    packed = torch.randint(0, 256, (N * K // 2,), dtype=torch.uint8, device=U.dev())
    scales = torch.rand(N // 16, K // 1024, 16, device=U.dev()).half()
    x = torch.randn(B, K, device=U.dev()).to(torch.bfloat16)
    y = torch.full((B, N), float("nan"), device=U.dev())
    rc = binding.lib.higgs_linear(d, x.data_ptr(), B, packed.data_ptr(), scales.data_ptr(), grid.data_ptr(), y.data_ptr(), hb.HIGGS_F32,
                                  None, 0, binding._stream())
    assert (hb.higgs_linear_launch_count(d, B) == 1) == one_launch
    assert rc == (hb.HIGGS_OK if one_launch else hb.HIGGS_ERR_INVALID_ARG)
    ref = hb.higgs_linear(d, x, packed, scales, grid, workspace=torch.empty(hb.higgs_workspace_bytes(d, hb.HIGGS_OP_LINEAR, B), dtype=torch.uint8, device=U.dev()))
    assert torch.equal(y, ref) if one_launch else y.isnan().all()
    assert torch.equal(hb.higgs_linear(d, x, packed, scales, grid), ref)
