"""A launch the runtime refuses reports its error and leaves none pending on the thread, so that
the next call's launches are judged by their own status.  The launch helper is compiled against a
fake runtime that refuses every launch the way the real one does (status returned and kept until
cudaGetLastError takes it); no GPU is involved."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FAKE = r"""
#include <cuda_runtime_api.h>
cudaError_t pending = cudaSuccess;
extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **) {
  return pending = cudaErrorStreamCaptureImplicit;
}
extern "C" cudaError_t cudaGetLastError() {
  const cudaError_t e = pending;
  pending = cudaSuccess;
  return e;
}
// what a compiled file calls at start-up (there are no kernels to register)
extern "C" void **__cudaRegisterFatBinary(void *) { return nullptr; }
extern "C" void __cudaRegisterFatBinaryEnd(void **) {}
extern "C" void __cudaUnregisterFatBinary(void **) {}
extern "C" char __cudaInitModule(void **) { return 0; }
"""
HARNESS = r"""
#include <cstdio>
#include "internal.h"
extern cudaError_t pending;
static void kern(int) {}
int main() {
  for (int dep = 0; dep < 2; dep++) {
    const cudaError_t e = fhe::launch_dep(dep != 0, kern, dim3(1), 32, 0, 0, 1);
    std::printf("%d ", e == cudaErrorStreamCaptureImplicit && pending == cudaSuccess);
  }
}
"""


def test_refused_launch_leaves_nothing_pending(tmp_path):
    from paper_2512_18345_gb300 import build
    try:
        nv = build.nvcc()
    except RuntimeError as e:
        pytest.skip(str(e))
    src, fake, exe = tmp_path / "harness.cu", tmp_path / "fake.cpp", tmp_path / "harness"
    src.write_text(HARNESS)
    fake.write_text(FAKE)
    cmd = [nv, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "--expt-relaxed-constexpr", "-cudart", "none",
           "-I", os.path.join(ROOT, "include"), "-I", build.CSRC, "-o", str(exe), str(src), str(fake)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split() == ["1", "1"]
