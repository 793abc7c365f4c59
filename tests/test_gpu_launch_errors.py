"""A launch that the runtime refuses on the host is reported once: it does not stay behind as the
last error of the thread, where the next launch check would find it."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

PKG = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_08733_gb300")


def test_refused_launch_leaves_no_error_behind(tmp_path):
    from paper_2002_08733_gb300 import build as B
    src = tmp_path / "launch.cu"
    src.write_text("""
#include "dgm_internal.h"
__global__ void nothing(int) {}
int main() {
    if (cudaFree(nullptr) != cudaSuccess) return 1;
    // more shared memory than a CTA may have: refused before anything reaches the GPU
    if (dgm::launch_ex(nothing, dim3(1), 32, size_t(1) << 30, 0, false, 1, 0) == cudaSuccess) return 2;
    if (cudaGetLastError() != cudaSuccess) return 3;
    if (dgm::launch_ex(nothing, dim3(1), 32, 0, 0, false, 1, 0) != cudaSuccess) return 4;
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : 5;
}
""")
    exe = str(tmp_path / "launch")
    subprocess.run([B.nvcc()] + B.ARCH + ["-std=c++17", "-I", B.INCLUDE, "-I", B.CSRC, str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0
