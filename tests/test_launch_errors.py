"""A launch that CUDA refuses is reported by the call that made it and by no
later one.  The launch helpers of common.cuh run here against a fake of the
runtime calls they make, whose launch fails when told to (no GPU)."""
import subprocess

from paper_2607_28897_gb300 import build

# The runtime's per-thread error state, and a launch that is refused on demand.
FAKE = r"""
int fake_last = 0, fake_refuse = 0;
extern "C" {
int cudaLaunchKernelExC(const void *, const void *, void **) {
  if (fake_refuse) fake_last = 1;
  return fake_refuse ? 1 : 0;
}
int cudaGetLastError(void) {
  const int e = fake_last;
  fake_last = 0;
  return e;
}
int cudaPeekAtLastError(void) { return fake_last; }
void **__cudaRegisterFatBinary(void *) {
  static void *h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
char __cudaInitModule(void **) { return 1; }
}
"""

SOURCE = r"""
#include "common.cuh"
#include <cstdio>

extern int fake_last, fake_refuse;
namespace bigint { void count_launch() {} }

static void kernel(int) {}
static int chain() { return bigint::chain_launch(true, kernel, 1u, 32u, 0, nullptr, 1); }
static cudaError_t failing() { fake_last = 1; return cudaErrorInvalidValue; }
static int tried() { BIGINT_CUDA_TRY(failing()); return BIGINT_OK; }

int main() {
  std::printf("%d ", chain());
  fake_refuse = 1;
  std::printf("%d ", chain());
  fake_refuse = 0;
  std::printf("%d ", chain());
  fake_last = 1;  // as a refused <<<>>> launch leaves it
  std::printf("%d ", bigint_launch_status());
  std::printf("%d ", bigint_launch_status());
  std::printf("%d ", tried());
  std::printf("%d\n", bigint_launch_status());
  return 0;
}
"""


def test_refused_launch_is_reported_once(tmp_path):
    src, fake, exe = tmp_path / "errors.cu", tmp_path / "fake.cpp", tmp_path / "errors"
    src.write_text(SOURCE)
    fake.write_text(FAKE)
    subprocess.run([build.nvcc()] + build.ARCH + ["-std=c++17", "-cudart", "none", "-I",
                   build.INCLUDE, "-I", build.CSRC, str(src), str(fake), "-o", str(exe)], check=True)
    got = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    assert got.split() == ["0", "-6", "0", "-6", "0", "-6", "0"]
