"""Search over one small codebook at the edges of its kernel: blocks of 16 codewords, the largest codebook of either type
(binary32 up to 1024 codewords, fp16 below 1024), the smallest of the kernels beyond (fp16: the tensor engine, binary32:
the FP32 engine), tiles of 32 and 64 targets, both splits of the targets."""
import os
import re

import numpy as np
import pytest

from paper_2405_14852_b200 import synth
from test_gpu_parity import check_encode

CASES = [
    (2, False, 1), (15, True, 31), (16, False, 32), (17, True, 33), (255, False, 64), (256, True, 65),
    (1000, True, 37887), (1023, False, 37888), (1023, True, 37889), (1024, False, 33), (1024, False, 37889),
    (1024, True, 37889), (1025, False, 37889), (300, False, 40000),
]


def test_the_cases_are_on_both_sides_of_the_rules():
    csrc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_14852_b200", "csrc")
    read = lambda name: open(os.path.join(csrc, name)).read()
    small = int(re.search(r"kM1SmallCodebook = (\d+);", read("pvt_internal.h")).group(1))
    tensor = int(re.search(r"kM1TensorCodebook = (\d+);", read("pvt_internal.h")).group(1))
    assert {small, small + 1} <= {K for K, f16, _ in CASES if not f16}
    assert {tensor - 1, tensor} <= {K for K, f16, _ in CASES if f16}


@pytest.mark.gpu
@pytest.mark.parametrize("K,f16,k", CASES)
def test_small_codebook_search_at_its_edges(K, f16, k):
    rows, cols = (128, 64) if k < 1000 else (640, 512)
    L = synth.make_layer(rows, cols, cfg=210, codebook_size=K, codebook_fp16=f16)
    idx = np.sort(np.random.default_rng(k).permutation(L.num_groups)[:k]).astype(np.uint32)
    check_encode(L, idx)
