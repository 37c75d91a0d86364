"""Search over one small codebook at the edges of its kernel: blocks of 16 codewords, the largest codebook of either type
(binary32 up to 1024 codewords, fp16 below 1024), the smallest of the kernels beyond (fp16: the tensor engine, binary32:
the FP32 engine), tiles of 32 and 64 targets, both splits of the targets.  A step over
every group is one kernel, with another for the weights of large layers: it leaves what the three calls leave."""
import os
import re

import numpy as np
import pytest
import torch

from paper_2405_14852_b200 import synth
from paper_2405_14852_b200.vstep import VStepLayer
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


@pytest.mark.gpu
@pytest.mark.parametrize("K,f16,rows,cols,out", [
    (2, False, 1, 16, "float32"),         # two groups
    (256, False, 256, 256, "float32"),
    (17, True, 33, 24, "float16"),        # a tile that is not full, rows that end inside a warp
    (1023, True, 129, 264, "float16"),
    (1024, False, 148, 2048, "float32"),  # two targets per team from here on
    (100, True, 641, 1000, "float16"),
    (300, False, 64, 72, None),           # no weights
    (200, True, 1000, 4000, "float16"),   # weights after the search: the least groups
    (200, False, 2000, 4000, "float32"),
    (64, False, 64, 72, "in place"),      # the weights take the place of W
])
def test_a_step_over_every_group_is_the_three_calls(K, f16, rows, cols, out):
    L = synth.make_layer(rows, cols, cfg=211, codebook_size=K, codebook_fp16=f16)
    if rows > 100:
        L.W[5, 16] = np.nan  # no codeword is nearest: the code stays, and the status says so
        L.codes[rows * cols // 8 - 1] = 255
    got = []
    for whole in (True, False):
        dev = VStepLayer.from_host(L)
        G = L.num_groups
        dev.reserve(G)
        idx = torch.full((G,), -1, dtype=torch.int32, device="cuda")
        W_hat = None
        if out == "in place":
            W_hat = dev.W
        elif out:
            W_hat = torch.full((rows, cols), 7.0, dtype=getattr(torch, out), device="cuda")
        if whole:
            dev.step(G, idx, W_hat)
        else:
            dev.select(G, idx)
            dev.encode(idx)
            if W_hat is not None:
                dev.dequant(W_hat)
        torch.cuda.synchronize()
        got.append((idx.cpu().numpy(), dev.codes.cpu().numpy(), dev.status(),
                    None if W_hat is None else W_hat.cpu().numpy().tobytes()))
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][0], np.arange(L.num_groups))
    assert np.array_equal(got[0][1], got[1][1])
    assert got[0][2:] == got[1][2:]
