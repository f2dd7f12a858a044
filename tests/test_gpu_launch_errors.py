"""A kernel launch that the runtime refuses, dependent or plain, leaves its error for the
check behind it, as the <<< >>> syntax does: a small CUDA program launches a CTA of
more threads than there can be, which the runtime refuses on the host."""
import os
import shutil
import subprocess

import pytest

from paper_1011_0911_gb300 import build_lib

pytestmark = pytest.mark.gpu

PROGRAM = """
#include <cstdio>
#include "lqcd_internal.cuh"
__global__ void k(int n) { after_previous(); }
int main()
{
    for (int pdl = 0; pdl < 2; pdl++) {
        launch_pdl(pdl, k, dim3(1), dim3(4096), (cudaStream_t)0, 1);
        const cudaError_t first = cudaGetLastError(), second = cudaGetLastError();
        printf("%d %d %d\\n", pdl, first != cudaSuccess, second != cudaSuccess);
    }
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="no nvcc")
def test_refused_launch_is_seen(tmp_path):
    src, exe = tmp_path / "launch.cu", tmp_path / "launch"
    src.write_text(PROGRAM)
    flags = [f for f in build_lib.FLAGS if f != "-lineinfo"]
    subprocess.run(["nvcc"] + build_lib.ARCH + flags + [str(src), "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, cwd=os.fspath(tmp_path)).stdout
    assert out.split("\n")[:2] == ["0 1 0", "1 1 0"]
