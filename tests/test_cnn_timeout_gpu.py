"""GEMM waits that run out: the MMA issuer stops after a few k-blocks, so the other
roles wait for stages that nothing frees. The product ends after one bounded wait,
reports it, leaves nothing in flight and the next product is right."""
import time

import pytest
import torch

pytestmark = pytest.mark.gpu


def _product(kind):
    """A product of one wave of CTAs and at least 9 k-blocks a CTA, as a function of the handle."""
    from paper_2003_06027_gb300 import learned as L

    g = torch.Generator().manual_seed(7)
    r = lambda *s: torch.randn(s, generator=g).cuda()
    if kind == "gemm":  # both operands by TMA
        a, b = (L.to_bf16(r(n, 640)) for n in (300, 48))
        return lambda h: L.gemm_bt(h, a, b, bias=torch.zeros(48, device="cuda"), relu=True)
    if kind == "wgrad":  # taps gathered M-major: 304 runs of 11 k-blocks
        x, dy, w = r(14, 3, 256, 256), r(16, 3, 256, 256), L.to_bf16(r(16, 14, 3, 3))
        y = torch.ones_like(dy)
        return lambda h: L.conv_backward(h, x, w, y, dy.clone(), 1, 1, True, need_dx=False)[1]
    # pixel pairs at stride 1 and 2, the tap table, the im2col matrix: 72 channels, 11 k-blocks
    C, H, W, s = {"pairs1": (72, 24, 32, 1), "pairs2": (72, 40, 64, 2), "table": (72, 24, 31, 1), "im2col": (72, 24, 32, 1)}[kind]
    x, w, b = r(C, 1, H, W), L.to_bf16(r(16, C, 3, 3)), r(16)

    def run(h):
        h.set_conv_gather(kind != "im2col")
        return L.conv_forward(h, x, w, b, s, s, True)

    return run


@pytest.mark.parametrize("limit", [0, 4, 5])
@pytest.mark.parametrize("kind", ["pairs1", "pairs2", "table", "im2col", "gemm", "wgrad"])
def test_wait_that_runs_out(fwi_lib, kind, limit):
    from paper_2003_06027_gb300 import fwi
    from paper_2003_06027_gb300 import learned as L

    h, run = L.Handle(0), _product(kind)
    want = run(h)
    h.check()
    h.selftest_issue_limit(limit)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    run(h)
    torch.cuda.synchronize()
    # the roles' waits run out together after 1 s; the waits for what is in flight add nothing to it
    assert time.perf_counter() - t0 < 3.0
    with pytest.raises(fwi.FwiError, match="timed out"):
        h.check()
    h.selftest_issue_limit(-1)
    assert torch.equal(run(h), want)
    h.check()


@pytest.mark.parametrize("kind", ["pairs1", "pairs2", "table", "im2col", "gemm", "wgrad"])
def test_output_of_a_timed_out_product_is_nan(fwi_lib, kind):
    # with the ReLU too, whose maximum of NaN and 0 is 0
    from paper_2003_06027_gb300 import fwi
    from paper_2003_06027_gb300 import learned as L

    h, run = L.Handle(0), _product(kind)
    h.selftest_issue_limit(3)
    assert bool(torch.isnan(run(h)).all())
    with pytest.raises(fwi.FwiError, match="timed out"):
        h.check()
