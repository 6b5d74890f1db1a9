"""A step's launch that fails leaves no error behind, which the next call would take for its own.  The launch has an
empty grid: the runtime refuses it on the host, and nothing reaches the GPU."""
import os
import subprocess

import pytest

from paper_1703_08015_gb300 import _build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "internal.h"
__global__ void k_nothing(int) {}
int main() {
    if (lbm::launch_chained(k_nothing, 0u, 32u, (cudaStream_t)0, 1) == cudaSuccess) return 1;
    return cudaGetLastError() == cudaSuccess ? 0 : 2;
}
"""


def test_failed_chained_launch_leaves_no_error(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")  # without one every call fails, and keeps failing
    nvcc = _build._nvcc()
    src, exe = tmp_path / "launch.cu", tmp_path / "launch"
    src.write_text(SOURCE)
    subprocess.run([nvcc, *_build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", _build.INCLUDE, "-I",
                    _build.CSRC, str(src), "-o", str(exe)], check=True, env=dict(os.environ))
    assert subprocess.run([str(exe)]).returncode == 0
