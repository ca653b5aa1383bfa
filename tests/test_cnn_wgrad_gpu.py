"""Weight gradients with the tap operand gathered inside the GEMM (pixel pairs,
14 channels a tile) equal those of the im2col matrix bit for bit: the same BF16
operands, the same k-blocks and splits."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# C, B, H, W, O, sh, sw: channel counts around a tile's 14 and its runs of 8 and 6; pixel counts off the
# 64-wide k-block; strides 1 and 2 across; widths that take the im2col path (odd, or odd pairs at stride 2)
SHAPES = [(1, 1, 2, 2, 1, 1, 1), (14, 1, 5, 6, 3, 1, 1), (15, 2, 7, 10, 17, 2, 1), (29, 1, 9, 34, 40, 4, 1),
          (8, 3, 3, 4, 256, 1, 1), (9, 1, 6, 8, 257, 2, 2), (16, 2, 11, 12, 24, 1, 2), (13, 1, 4, 7, 5, 1, 1),
          (6, 2, 5, 6, 9, 2, 2), (64, 1, 33, 30, 32, 1, 1)]


@pytest.mark.parametrize("shape", SHAPES, ids=["x".join(map(str, s)) for s in SHAPES])
def test_gathered_weight_gradient_equals_im2col(fwi_lib, shape):
    import torch

    from paper_2003_06027_gb300 import learned as L

    C, B, H, W, O, sh, sw = shape
    g = torch.Generator().manual_seed(C * 100 + W)
    x = torch.randn((C, B, H, W), generator=g).cuda()
    wb = L.to_bf16((torch.randn((O, C, 3, 3), generator=g) * 0.3).cuda())
    b = torch.zeros(O, device="cuda")
    dy0 = torch.randn((O, B, L.conv_out(H, sh), L.conv_out(W, sw)), generator=g).cuda()
    out = []
    for on in (True, False):
        h = L.Handle(0)
        h.set_conv_gather(on)
        y = L.conv_forward(h, x, wb, b, sh, sw, True)
        out.append((y, *L.conv_backward(h, x, wb, y, dy0.clone(), sh, sw, True)))
        h.check()
    for p, q in zip(*out):
        assert torch.equal(p, q)
    # and the sum itself, on the BF16-rounded operands in FP64: FP32 accumulation of at most 1e3 products
    r = lambda t: t.bfloat16().double()
    dyr = r(torch.where(out[0][0] > 0, dy0, torch.zeros_like(dy0))).transpose(0, 1)
    xr = torch.nn.functional.pad(r(x).transpose(0, 1), (1, 1, 1, 1))
    ref = torch.stack([torch.einsum("bohw,bchw->oc", dyr, xr[:, :, p:p + sh * dyr.shape[2]:sh, q:q + sw * dyr.shape[3]:sw][:, :, :dyr.shape[2], :dyr.shape[3]])
                       for p in range(3) for q in range(3)], -1).reshape(O, C, 3, 3)
    assert float((out[0][2].double() - ref).norm()) <= 1e-5 * float(ref.norm()) + 1e-30
