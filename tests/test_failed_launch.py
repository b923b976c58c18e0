"""A launch that the runtime refuses is reported by the call, and is not left behind in the thread, where the next library that
asks for the last error takes it for its own.  On a stand-in for the CUDA runtime: without a driver the real one has an error at all
times."""
import shutil
import subprocess

import pytest

from paper_2605_06665_b200 import build as builder

RUNTIME = r"""
int last, capture_answer, launch_answer;
extern "C" {
int cudaStreamIsCapturing(void*, int* state) {
  *state = 0;
  return capture_answer != 0 ? last = capture_answer : 0;
}
int cudaLaunchKernelExC(const void*, const void*, void**) { return launch_answer != 0 ? last = launch_answer : 0; }
int cudaGetLastError() { const int e = last; last = 0; return e; }
const char* cudaGetErrorString(int) { return ""; }
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
}
"""
CALLER = r"""
#include <cstdio>
#include "common.cuh"
extern int last, capture_answer, launch_answer;
namespace unipool { void set_error(const char*, ...) {} }
static void kern(int) {}
static int launch() {
  UP_KERNEL(kern, 1, 32, 0, nullptr, 0);
  return UNIPOOL_OK;
}
int main() {
  const int answers[3][2] = {{0, 0}, {0, cudaErrorInvalidConfiguration}, {cudaErrorStreamCaptureImplicit, 0}};
  for (auto& a : answers) {
    capture_answer = a[0];
    launch_answer = a[1];
    const int rc = launch();
    printf("%d %d ", rc, last);
    last = 0;
  }
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="needs nvcc")
def test_failed_launch_leaves_no_error(tmp_path):
    (tmp_path / "launch.cu").write_text(CALLER)
    (tmp_path / "runtime.cpp").write_text(RUNTIME)
    exe = str(tmp_path / "launch")
    flags = [f for f in builder.NVCC_FLAGS if f not in ("-Xcompiler", "-fPIC")]
    subprocess.run(["nvcc"] + flags + ["-cudart", "none", "launch.cu", "runtime.cpp", "-o", exe], cwd=tmp_path, check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert [int(v) for v in out] == [0, 0, -4, 0, -4, 0]
