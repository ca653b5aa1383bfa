"""Products of different shared-memory sizes from two host threads, each with a handle
and a stream of its own: no launch of one fails for what the other has just launched."""
import ctypes
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


def _calls(L, K, N, n, fails):
    """n products of 128 rows with K taps and N columns, issued back to back."""
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        h = L.Handle(0)
        a, b = (torch.zeros((r, K), dtype=torch.int16, device="cuda") for r in (128, N))
        out = torch.empty((N, 128), device="cuda")
        f, P = L._lib().fwi_cnn_gemm_bt, ctypes.c_void_p
        args = (h.h, P(a.data_ptr()), K, P(b.data_ptr()), K, 128, N, K, P(out.data_ptr()), 128, None, 0, 1,
                P(s.cuda_stream))
        bad = 0
        for _ in range(n):
            bad += f(*args) != 0
        s.synchronize()
        h.check()
    fails.append(bad)


def test_threads_with_products_of_different_sizes(fwi_lib):
    from paper_2003_06027_gb300 import learned as L

    fails = []
    # 1 stage of 16 columns against 4 of 256
    th = [threading.Thread(target=_calls, args=(L, K, N, 40000, fails)) for K, N in ((8, 16), (256, 256))]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert fails == [0, 0]
