"""A refused kernel launch is reported by its own call and by no later one.

launch_kernel (dkv_internal.h) is linked with fakes of the two runtime calls it makes:
a launch that the fake refuses must come back as the return value and leave no pending
error, which the next call that asks cudaGetLastError() would report as its own.
"""
import os
import subprocess

import pytest

from paper_2608_27922_gb300 import build as B

FAKES = r"""
int pending = 0, refuse = 0;
extern "C" int cudaLaunchKernelExC(const void*, const void*, void**) {
  if (refuse) pending = refuse;
  return refuse;
}
extern "C" int cudaGetLastError(void) {
  const int e = pending;
  pending = 0;
  return e;
}
"""
SRC = r"""
#include "dkv_internal.h"
extern int pending, refuse;
static void k(int) {}
int main() {
  const int cases[][2] = {{1, 0}, {1, 1}, {4, 0}, {4, 1}};   // cluster, after
  for (int error : {0, (int)cudaErrorInvalidConfiguration})
    for (auto& c : cases) {
      refuse = error;
      if ((int)dkv::launch_kernel(k, dim3(4), 32, 0, c[0], c[1] != 0, (cudaStream_t)0, 1) != error) return 1;
      if (pending != 0) return 2;
    }
  return 0;
}
"""


def test_a_refused_launch_leaves_no_pending_error(tmp_path):
    try:
        nvcc = B.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    src, fakes, exe = tmp_path / "launch.cu", tmp_path / "fakes.cpp", tmp_path / "launch"
    src.write_text(SRC)
    fakes.write_text(FAKES)
    subprocess.check_call([nvcc, *B.ARCH, "-std=c++17", "-cudart", "shared", "-I", B.ROOT + "/include", "-I", B.CSRC,
                           str(src), str(fakes), "-o", str(exe),
                           "-Xlinker", "-rpath=" + os.path.join(os.path.dirname(os.path.dirname(nvcc)), "lib64")])
    assert subprocess.run([str(exe)]).returncode == 0
