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


@pytest.mark.parametrize("B", [1, 2, 5, 16, 40])
@pytest.mark.parametrize("N,K", [(1024, 1024), (2048, 2048), (8192, 2048)])
def test_a_chain_reads_what_the_product_before_it_wrote(N, K, B):
    """Every kernel starts while the one before it runs; activations that it has just written, over older ones that were read a moment
    ago, are what the next product sees."""
    g = torch.Generator(device="cuda").manual_seed(B)
    _, grid = U.grid32(2, 256)
    down, up = hb.make_desc(2, 256, K, N, 7), hb.make_desc(2, 256, N, K, 8)
    weights = [(torch.randint(0, 256, (N * K // 2,), dtype=torch.uint8, device="cuda", generator=g),
                (torch.rand(N * K // 1024, device="cuda", generator=g) * (2.0 / inputs) ** 0.5).half()) for inputs in (K, N)]
    x0 = torch.randn(B, K, device="cuda", generator=g).to(torch.bfloat16)
    ws = torch.empty(max(hb.higgs_workspace_bytes(d, hb.HIGGS_OP_LINEAR, B) for d in (up, down)), dtype=torch.uint8, device="cuda")

    def run(steps, wait):
        x, h, seen = x0.clone(), torch.zeros(B, N, dtype=torch.bfloat16, device="cuda"), []
        for _ in range(steps):
            hb.higgs_linear(up, x, *weights[0], grid, workspace=ws, y=h)
            if wait:
                torch.cuda.synchronize()
            hb.higgs_linear(down, h, *weights[1], grid, workspace=ws, y=x)
            if wait:
                torch.cuda.synchronize()
                seen.append(x.clone())
        return seen if wait else x

    seen = run(12, True)
    assert torch.isfinite(seen[-1].float()).all() and seen[-1].float().abs().max() > 1e-3
    if any(hb.higgs_linear_uses_atomics(d, B) for d in (up, down)):
        pytest.skip("K ranges that meet in atomics: no two runs are alike")
    for steps in (1, 2, 5, 12):
        assert torch.equal(run(steps, False), seen[steps - 1])
