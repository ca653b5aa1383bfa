"""A step launch that the runtime refuses is reported once: the launch after it is
judged by itself."""
import os
import subprocess

import pytest

from paper_2003_06027_gb300 import build

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cstdio>
#include "tma.cuh"
__global__ void k(int*) {}
int main() {
  int* none = nullptr;
  const cudaError_t refused = fwi::launch_step(k, 1, 0, 32, 0, 0, none);  // an empty grid: refused on the host
  k<<<1, 32>>>(none);
  printf("%d %d %d\n", refused != cudaSuccess, (int)cudaGetLastError(), (int)cudaDeviceSynchronize());
}
"""


def test_refused_launch_is_reported_once(tmp_path):
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-I", build.CSRC, "-I", os.path.join(build.ROOT, "include"),
                    "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split() == ["1", "0", "0"]
