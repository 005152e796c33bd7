"""The rotation with four warps per group (layers that leave SMs free) against the one for large layers: the same bits."""
import pytest
import torch

import paper_2411_17525_b200 as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,K", [(1, 1024), (1, 8192), (3, 3072), (5, 2048), (16, 1024), (8, 4096)])
def test_small_batch(B, K):
    x = torch.randn(B, K, device="cuda", generator=torch.Generator(device="cuda").manual_seed(B)).to(torch.bfloat16)
    small, large = (hb.higgs_rotate_activations(hb.make_desc(2, 256, N, K, 99), x) for N in (16, 28672))
    assert torch.equal(small, large)


@pytest.mark.parametrize("B,K", [(17, 1024), (31, 4096), (33, 3072), (100, 2048), (144, 1024), (200, 1024)])
def test_blocked_layout(B, K):
    """Padding tokens are zeros whatever the buffer held."""
    x = torch.randn(B, K, device="cuda", generator=torch.Generator(device="cuda").manual_seed(B)).to(torch.bfloat16)
    got = []
    for N in (128, 28672):
        d = hb.make_desc(2, 256, N, K, 98)
        out = torch.full((hb.higgs_rotated_bytes(d, B) // 2,), float("nan"), dtype=torch.float16, device="cuda")
        hb.higgs_rotate_activations(d, x, out)
        got.append(out)
    assert torch.equal(*got)
