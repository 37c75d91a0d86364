"""Host rules of the library in small host programs (no GPU).  Setting a kernel up for large shared memory asks the driver once
per kernel, however many kernels share a signature (the CUDA calls are counted instead of made); a step dequantises ahead of its
search where that was measured to be no slower."""
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


RULE = r"""
#include <cstdio>
#include <type_traits>
#include "pvt_internal.h"
// weights beside the selection: by the plain norms, no other keys
static_assert(!std::is_invocable_v<decltype(pvt::launch_select_keyed), const pvt_layer&, uint64_t, uint64_t, uint32_t*,
                                   void*, int, cudaStream_t, int, float*, uint64_t, void*, int32_t>);
int main() {
  int rows, cols, M, K, dg, f16, out_f16, part;
  while (std::scanf("%d %d %d %d %d %d %d %d", &rows, &cols, &M, &K, &dg, &f16, &out_f16, &part) == 8) {
    pvt_layer L = {};
    L.group_dim = dg, L.num_codebooks = M, L.codebook_size = K, L.codebook_dtype = f16 ? PVT_F16 : PVT_F32;
    const uint64_t G = (uint64_t)rows * cols / dg;
    const int32_t out = out_f16 ? PVT_F16 : PVT_F32;
    std::printf("%d ", (int)(part == 1 ? pvt::step_weights_after(L, G, out) : pvt::step_dequant_first(L, G / part, G, out)));
  }
}
"""


def run(tmp_path, program, given=""):
    src, exe = tmp_path / "program.cu", tmp_path / "program"
    src.write_text(program)
    subprocess.run(["nvcc", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2405_14852_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True, input=given).stdout


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="no nvcc")
def test_the_driver_is_asked_once_per_kernel_and_device(tmp_path):
    assert int(run(tmp_path, PROGRAM)) == 2 * 12 + 12


# rows, cols, codebooks, codewords, group, fp16 codebook, fp16 weights, one group in so many
SLOWER_FIRST = [
    (1024, 1024, 3, 256, 8, 0, 1, 100), (1024, 1536, 3, 256, 8, 0, 1, 200), (1024, 1536, 4, 256, 8, 0, 1, 100),
    (1024, 1024, 4, 256, 8, 1, 1, 100), (8192, 8192, 4, 256, 8, 1, 1, 32), (11008, 4096, 4, 256, 8, 1, 1, 12),
    (28672, 8192, 1, 512, 8, 1, 1, 16), (28672, 8192, 1, 256, 8, 0, 0, 32), (28672, 8192, 1, 4096, 8, 1, 0, 12),
    (8192, 8192, 2, 256, 8, 1, 0, 8), (4096, 4096, 1, 65536, 8, 1, 0, 4), (28672, 8192, 4, 256, 8, 1, 0, 100),
]
FASTER_FIRST = [
    (4096, 4096, 1, 65536, 8, 1, 0, 100), (11008, 4096, 2, 256, 8, 1, 0, 100), (11008, 4096, 3, 256, 8, 1, 1, 100),
    (4096, 4096, 1, 65536, 16, 1, 1, 100), (28672, 8192, 1, 65536, 8, 1, 1, 16), (28672, 8192, 2, 256, 8, 0, 1, 32),
    (8192, 8192, 2, 256, 8, 0, 1, 8), (28672, 8192, 1, 256, 8, 0, 1, 32), (28672, 8192, 1, 512, 8, 1, 1, 200),
    (11008, 4096, 4, 256, 8, 1, 1, 100), (256, 512, 1, 256, 8, 1, 0, 100), (512, 1024, 2, 256, 8, 0, 1, 48),
]


# the same of steps over every group: weights from the search itself, and from a kernel after it
FASTER_INSIDE = [(256, 256, 1, 256, 8, 0, 0, 1), (1024, 2048, 1, 256, 8, 1, 1, 1), (4096, 4096, 1, 1000, 8, 1, 0, 1),
                 (2048, 2048, 1, 4, 8, 1, 0, 1)]
FASTER_AFTER = [(2048, 2048, 1, 4, 8, 1, 1, 1), (4096, 4096, 1, 256, 8, 1, 1, 1), (28672, 8192, 1, 1000, 8, 1, 1, 1),
                (4096, 4096, 1, 256, 8, 0, 0, 1), (28672, 8192, 1, 512, 8, 1, 0, 1)]


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="no nvcc")
def test_weights_of_all_groups_come_from_the_faster_kernel(tmp_path):
    given = "\n".join(" ".join(map(str, case)) for case in FASTER_INSIDE + FASTER_AFTER)
    got = [int(x) for x in run(tmp_path, RULE, given).split()]
    assert got == [0] * len(FASTER_INSIDE) + [1] * len(FASTER_AFTER)


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="no nvcc")
def test_weights_are_written_ahead_of_the_search_where_that_is_no_slower(tmp_path):
    given = "\n".join(" ".join(map(str, case)) for case in SLOWER_FIRST + FASTER_FIRST)
    got = [int(x) for x in run(tmp_path, RULE, given).split()]
    assert got == [0] * len(SLOWER_FIRST) + [1] * len(FASTER_FIRST)
