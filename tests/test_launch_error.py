"""A refused launch leaves the runtime's last error clear (no GPU needed).

The launch helper is compiled against a runtime whose launch call fails: its
status comes back, and the caller's next look at the last error finds none."""
import os
import shutil
import subprocess

import pytest

from paper_1103_0066_gb300 import build

PROGRAM = r"""
#include <cuda_runtime.h>
#include "fem_internal.h"
static cudaError_t last = cudaSuccess, next = cudaSuccess;
extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) {
  if (next != cudaSuccess) last = next;
  return next;
}
extern "C" cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
static void kern(int) {}
int main() {
  next = cudaErrorInvalidConfiguration;
  if (fem::launch_chained(kern, 1u, 32u, 0, nullptr, 7) != cudaErrorInvalidConfiguration) return 1;
  if (last != cudaSuccess) return 2;
  next = cudaSuccess;
  return fem::launch_chained(kern, 1u, 32u, 0, nullptr, 7) == cudaSuccess ? 0 : 3;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host compiler")
def test_refused_launch_clears_the_last_error(tmp_path):
    cuda = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    (tmp_path / "t.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", cuda, "-I", build.CSRC, "-I", build.INCLUDE, str(tmp_path / "t.cpp"),
                    "-o", str(tmp_path / "t")], check=True)
    assert subprocess.run([str(tmp_path / "t")]).returncode == 0
