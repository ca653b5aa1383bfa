"""The pair-gathering convolution products against the materialised operand: more
tiles than persistent CTAs, runs of 8 channels that do not fill the gathering groups
evenly, channel tails, two column tiles, both horizontal strides, odd heights."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,B,H,W,O,sh,sw", [
    (8, 1, 201, 200, 16, 1, 1),      # 315 tiles of 128 pixels, two runs a tile
    (40, 3, 101, 136, 24, 1, 1),     # five runs over four groups, 323 tiles
    (13, 2, 57, 90, 9, 1, 1),        # a channel tail in the last run
    (9, 1, 129, 64, 272, 2, 2),      # two column tiles, one channel in the last run
    (24, 1, 3, 2, 8, 1, 1),          # less than one tile
    (72, 1, 403, 196, 8, 2, 2),      # nine runs, more k-blocks than stages
])
def test_pairs_equal_im2col(C, B, H, W, O, sh, sw):
    # the same BF16 operands in the same order of accumulation: equal bit for bit
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
