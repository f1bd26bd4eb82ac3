"""A launch that the CUDA runtime refuses is reported by the call that made it
and leaves no error behind for the check of a later, valid call (an empty grid,
which the runtime refuses on the host)."""
import os
import shutil
import subprocess

import pytest

from paper_2109_14704_gb300.build import ARCH, CSRC

pytestmark = pytest.mark.gpu      # without a driver every call of the runtime fails

PROGRAM = r"""
#include <cstdio>
#include "launch.h"
__global__ void k(int) { he::stream_order(); }
int main()
{
    cudaGetLastError();
    const cudaError_t e = he::launch_k(k, 0, 32, 0, 1, (cudaStream_t)0, 1);
    std::printf("%d %d\n", e != cudaSuccess, cudaPeekAtLastError() != cudaSuccess);
}
"""


def test_a_refused_launch_leaves_no_error_behind(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    (tmp_path / "p.cu").write_text(PROGRAM)
    exe = str(tmp_path / "p")
    subprocess.run([nvcc, *ARCH, "-std=c++17", "-I", CSRC, str(tmp_path / "p.cu"), "-o", exe], check=True,
                   capture_output=True, timeout=300)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout.split()
    assert out == ["1", "0"]
