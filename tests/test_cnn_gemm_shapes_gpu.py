"""The TMA-staged GEMM at the edges of its stage ring (1 to 5 k-blocks, so 1 to 4
stages and several CTAs per SM) and of its column tiles (one, two and three)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [
    (128, 16, 8), (1000, 257, 64), (4099, 288, 65), (2500, 300, 128), (777, 576, 192), (130, 48, 256), (300, 512, 320),
])
def test_gemm_bt(M, N, K):
    from paper_2003_06027_gb300 import learned as L

    g = torch.Generator().manual_seed(M + N + K)
    ld = (K + 7) // 8 * 8
    a, b = torch.randn((M, ld), generator=g).bfloat16(), torch.randn((N, ld), generator=g).bfloat16()
    h = L.Handle(0)
    out = L.gemm_bt(h, a.view(torch.int16).cuda()[:, :K], b.view(torch.int16).cuda()[:, :K]).cpu().double()
    h.check()
    a, b = a[:, :K].double(), b[:, :K].double()
    # FP32 accumulation of K exact products, each addition rounded or truncated at 2^-22 of the sum of magnitudes
    tol = K * 2.0 ** -22 * (b.abs() @ a.abs().T)
    assert bool(((out - b @ a.T).abs() <= tol).all())
