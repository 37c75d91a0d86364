"""Setting a kernel up for large shared memory asks the driver once per kernel, however many kernels share a signature: the
library's own helper in a small host program whose CUDA calls are counted instead of made (no GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <utility>
#include <cuda_runtime.h>
static int asked = 0;
#define cudaFuncGetAttributes(fa, kernel) ((void)(kernel), (fa)->sharedSizeBytes = 0, ++asked, cudaSuccess)
#define cudaFuncSetAttribute(kernel, what, value) ((void)(kernel), (void)(value), cudaSuccess)
#include "pvt_internal.h"
static int device = 0;
int pvt::device_slot() { return device; }
namespace {
template <int N>
__global__ void some_kernel(int* p) { *p = N; }
template <int... N>
void all(std::integer_sequence<int, N...>) { (void)std::initializer_list<int>{(int)pvt::allow_smem<some_kernel<N>>()...}; }
}
int main() {
  for (device = 0; device < 2; ++device)
    for (int round = 0; round < 3; ++round) all(std::make_integer_sequence<int, 12>());
  device = -1;  // a device beyond the table: asked every time
  all(std::make_integer_sequence<int, 12>());
  std::printf("%d\n", asked);
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="no nvcc")
def test_the_driver_is_asked_once_per_kernel_and_device(tmp_path):
    src, exe = tmp_path / "setup.cu", tmp_path / "setup"
    src.write_text(PROGRAM)
    subprocess.run(["nvcc", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2405_14852_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    assert int(out) == 2 * 12 + 12
