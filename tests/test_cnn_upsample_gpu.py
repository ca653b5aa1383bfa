"""Upsampling and its transpose around the launcher's block sizes (64, 128 and 256
threads: a block for each SM) and walks of several items a thread, odd and even rows."""
import pytest
import torch

pytestmark = pytest.mark.gpu


# items (pairs of even rows): 1; 9727, 9728 and 38 911, 38 912 (152 x 64 and x 256); more than the largest grid
@pytest.mark.parametrize("C,B,H,W", [(1, 1, 1, 1), (1, 1, 71, 137), (1, 1, 64, 304), (1, 1, 167, 233), (2, 1, 128, 304),
                                     (19, 8, 64, 257), (40, 2, 125, 252)])
def test_upsample_and_transpose(fwi_lib, C, B, H, W):
    from paper_2003_06027_gb300 import learned as L

    g = torch.Generator().manual_seed(H * W)
    x = torch.randn((C, B, H, W), generator=g).cuda()
    y = L.upsample2(x)
    assert torch.equal(y, x.repeat_interleave(2, 2).repeat_interleave(2, 3))
    dy = torch.randn(y.shape, generator=g).cuda()
    q = dy.view(C, B, H, 2, W, 2)
    want = (q[:, :, :, 0, :, 0] + q[:, :, :, 0, :, 1]) + (q[:, :, :, 1, :, 0] + q[:, :, :, 1, :, 1])
    assert torch.equal(L.upsample2_backward(dy), want)
