"""A launch that fails is reported once: the helpers every kernel is launched with (csrc/lg_host.h) leave no error behind in
the runtime, where a later call that succeeded would find it.  Compiled for the host against a stand-in for the runtime's
launch functions; no GPU."""
import os
import shutil
import subprocess

import pytest

from paper_2410_01485_b200 import build

SOURCE = r"""
#define __forceinline__ inline
#include <cuda_runtime.h>
template <typename T> static cudaError_t cudaFuncSetAttribute(T* f, cudaFuncAttribute a, int v) { return ::cudaFuncSetAttribute((const void*)f, a, v); }
#include "lg_host.h"
#include <cstdio>
static cudaError_t last = cudaSuccess;
static int launch_failures = 0, attribute_failures = 0, launched = 0;
static cudaError_t result(int& failures) {
  if (failures == 0) return cudaSuccess;
  --failures;
  return last = cudaErrorInvalidValue;
}
extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) { return result(launch_failures); }
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return result(attribute_failures); }
extern "C" cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
extern "C" cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
namespace lg { void note_launch() { ++launched; } }
static void kernel(int) {}
int main() {
  static std::atomic<bool> allowed[lg::kMaxDevices];
  auto plain = [](int fail) { launch_failures = fail; return lg::launch_kernel(true, kernel, dim3(1), 32, 0, nullptr, 3); };
  auto big = [](int fail, int attr) {
    launch_failures = fail; attribute_failures = attr;
    return lg::launch_big_smem(false, allowed, kernel, dim3(1), 32, 1 << 17, nullptr, 3);
  };
  int bad = 0;
  auto expect = [&](cudaError_t got, bool ok, int n) { bad += ((got == cudaSuccess) != ok) + (last != cudaSuccess) + (launched != n); };
  expect(plain(0), true, 1);
  expect(plain(1), false, 1);
  expect(big(0, 1), false, 1);           // the attribute is refused
  expect(big(1, 0), false, 1);           // the first launch on a device fails
  expect(big(0, 0), true, 2);
  expect(big(1, 0), true, 3);            // the device has forgotten the attribute: set again, launched again
  expect(big(2, 0), false, 3);
  expect(big(1, 1), false, 3);
  std::printf("%d\n", bad);
  return bad;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host compiler")
def test_a_failed_launch_leaves_no_error_behind(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", build.CSRC, "-I", os.path.join(cuda, "include"), str(src), "-o",
                    str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.stdout.split() == ["0"] and out.returncode == 0
