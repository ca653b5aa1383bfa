"""Convolution products on both sides of the line between the pair-gathering kernel and
the tap table, and channel tails of the former: the same bits as the im2col matrix."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,B,H,W,O,sh,sw", [
    (31, 1, 152, 128, 16, 1, 1),   # 152 tiles, one for each SM: the table up to 31 channels
    (32, 1, 152, 128, 16, 1, 1),
    (11, 1, 304, 128, 80, 1, 1),   # one tile for each CTA, two an SM: the table up to 11
    (12, 1, 304, 128, 80, 1, 1),
    (11, 1, 153, 128, 96, 1, 1),   # one CTA an SM: two tiles for one of them
    (8, 1, 305, 128, 16, 1, 1),
    (7, 1, 305, 128, 16, 1, 1),    # too few channels for pairs
    (13, 2, 115, 180, 9, 1, 1),    # a channel tail in the last run, 324 tiles
    (9, 1, 300, 136, 272, 2, 2),   # stride 2, two column tiles, one channel in the last run
    (36, 1, 57, 90, 24, 1, 1),     # one tile a CTA, a tail of four channels
    (33, 2, 30, 32, 17, 2, 2),
])
def test_both_sides_equal_im2col(fwi_lib, C, B, H, W, O, sh, sw):
    from paper_2003_06027_gb300 import learned as L

    g = torch.Generator().manual_seed(C * H + O)
    x = torch.randn((C, B, H, W), generator=g).cuda()
    wb = L.to_bf16(torch.randn((O, C * 9), generator=g).cuda())
    b = torch.randn(O, generator=g).cuda()
    h = L.Handle(0)
    ys = []
    for gather in (False, True, True):
        h.set_conv_gather(gather)
        ys.append(L.conv_forward(h, x, wb, b, sh, sw, True))
        h.check()
    assert torch.equal(ys[0], ys[1]) and torch.equal(ys[1], ys[2])
