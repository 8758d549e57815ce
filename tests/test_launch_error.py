"""A chained launch that the runtime refuses reports its error to the caller and
leaves none behind for the next CUDA call of the program to trip over."""
import subprocess

import pytest

from paper_2608_09703_gb300 import build as mbuild

SOURCE = """
#include "mls_kernels.h"
__global__ void kernel(int) {}
int main() {
  // more threads than a block may have: the runtime refuses it on the host
  const cudaError_t e = mls::launch_chained(kernel, dim3(1), dim3(4096), 0, nullptr, 1);
  return e != cudaSuccess && cudaPeekAtLastError() == cudaSuccess ? 0 : 1;
}
"""


@pytest.mark.gpu  # without a device the runtime's own error never clears
def test_refused_launch_leaves_no_error(tmp_path):
    src, exe = tmp_path / "refused.cu", tmp_path / "refused"
    src.write_text(SOURCE)
    subprocess.run([mbuild.nvcc(), *mbuild.ARCH, "-std=c++17", "-I", mbuild.CSRC,
                    "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
