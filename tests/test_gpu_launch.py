"""A kernel launch that the runtime refuses is reported once: it leaves no error behind that the next
search, which reads the runtime's last error after its own launches, would take for its own."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1804_09996_gb300", "csrc")
PROGRAM = r"""
#include <cstdio>
#include "lc_walk.cuh"
__global__ void one(int *p) { *p = 1; }
int main()
{
    int *p = nullptr;
    if (cudaMalloc(&p, 4) != cudaSuccess) return 2;
    for (bool pdl : {false, true}) {
        // more threads than a block can have: refused before anything reaches the device
        if (lc::launch(one, 1, 4096, 0, (cudaStream_t)0, pdl, p) == cudaSuccess) return 3;
        if (cudaGetLastError() != cudaSuccess) return 4;
        if (lc::launch(one, 1, 32, 0, (cudaStream_t)0, pdl, p) != cudaSuccess) return 5;
    }
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : 6;
}
"""


@pytest.mark.gpu
def test_refused_launch_leaves_no_error(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src, exe = tmp_path / "launch.cu", tmp_path / "launch"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    assert subprocess.run([str(exe)], timeout=60).returncode == 0
