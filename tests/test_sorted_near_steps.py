"""The steps nearest to a step, as the search in spatial order ranks them: whatever the boxes, each of the first ranks has
exactly one step (a rank without a step would be a place of the list that nobody writes).  The kernel's own key in a small
host program (no GPU)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include <vector>
#include "pvt_encode_m1_sorted.cuh"
using namespace pvt::m1;
// stdin: the number of steps, a distance for each pair of them; stdout: row by row the step of each rank (65535: none)
int main() {
  uint32_t n = 0;
  if (std::fread(&n, 4, 1, stdin) != 1) return 1;
  std::vector<float> d((size_t)n * n);
  if (std::fread(d.data(), 4, d.size(), stdin) != d.size()) return 1;
  for (uint32_t s = 0; s < n; ++s) {
    uint32_t key[kSortedSteps];
    for (uint32_t i = 0; i < kSortedSteps; ++i) {
      uint32_t bits = 0x7f800000u;
      if (i < n) std::memcpy(&bits, &d[(size_t)s * n + i], 4);
      key[i] = near_key(bits, i, s);
    }
    std::vector<uint16_t> near(kSortedNear, 65535);
    for (uint32_t i = 0; i < n; ++i) {
      uint32_t rank = 0;
      for (uint32_t q = 0; q < kSortedSteps; ++q) rank += key[q] < key[i];
      if (rank < kSortedNear) near[rank] = (uint16_t)i;
    }
    std::fwrite(near.data(), 2, near.size(), stdout);
  }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("nvcc") is None:
        pytest.skip("no nvcc")
    at = tmp_path_factory.mktemp("near")
    (at / "near.cu").write_text(PROGRAM)
    subprocess.run(["nvcc", "-O2", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I",
                    os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2405_14852_b200", "csrc"), "-o",
                    str(at / "near"), str(at / "near.cu")], check=True)
    return str(at / "near")


def distances(centres):
    return ((centres[:, None].astype(np.float32) - centres[None].astype(np.float32)) ** 2).sum(-1, dtype=np.float32)


def boxes(kind):
    rng = np.random.default_rng(3)
    if kind == "one codeword":  # 60000 codewords: all centres are the same
        return distances(np.full((469, 8), 0.25))
    c = rng.normal(size=(512 if kind != "fewest steps" else 257, 8))
    if kind == "first two":
        c[1] = c[0]
    elif kind == "copies":
        c = np.tile(c[:2], (256, 1))
    elif kind == "half of them":  # dead codewords in many cells
        c[::2] = 0
    d = distances(c)
    if kind == "empty boxes":
        d[5::7] = d[:, 5::7] = np.inf
    return d


@pytest.mark.parametrize("kind", ["one codeword", "first two", "copies", "half of them", "empty boxes", "fewest steps",
                                  "random"])
def test_every_rank_has_a_step(program, kind):
    d = boxes(kind)
    n = len(d)
    out = subprocess.run([program], input=np.uint32(n).tobytes() + d.tobytes(), check=True, capture_output=True).stdout
    near = np.frombuffer(out, np.uint16).reshape(n, 32).astype(np.int64)
    assert near.max() < n
    assert (np.sort(near, 1)[:, 1:] > np.sort(near, 1)[:, :-1]).all()  # 32 different steps
    assert (near[:, 0] == np.arange(n)).all()
    if kind == "random":
        order = np.argsort(np.where(np.eye(n, dtype=bool), -1, d), 1, kind="stable")[:, :32]
        assert (near == order).mean() > 0.99  # (a distance loses its last nine bits)
