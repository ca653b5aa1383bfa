"""Split products: the partials of every number of splits are added in order."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("splits", [2, 3, 4, 5, 6, 7, 8, 9, 12, 15, 16, 17])
def test_partials_are_added_in_order(fwi_lib, splits):
    from paper_2003_06027_gb300 import learned as L

    M, N, K = 131, 17, 64 * splits
    g = torch.Generator().manual_seed(splits)
    a, b = (L.to_bf16(torch.randn((r, K), generator=g).cuda()) for r in (M, N))
    h = L.Handle(0)
    want = None
    for k in range(0, K, 64):  # one k-block a split
        p = L.gemm_bt(h, a[:, k:k + 64], b[:, k:k + 64])
        want = p if want is None else want + p
    assert torch.equal(L.gemm_bt(h, a, b, splits=splits), want)
    h.check()
