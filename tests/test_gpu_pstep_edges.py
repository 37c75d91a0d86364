"""Gradients of the P step where the accumulation changes: sums in shared memory against sums in the L2, tiles and
warps that are not full, rows that end inside a warp, an update matrix on a 16-byte boundary only."""
import os
import re

import numpy as np
import pytest
import torch

from oracle import pvt_oracle as oracle
from paper_2405_14852_b200 import binding as B


CASES = [
    (1, 1024, True, 41, 25, 8, 0),     # the largest codebook summed in shared memory; 1025 groups: one in the last tile
    (1, 1024, False, 300, 129, 8, 4),
    (4, 256, True, 41, 25, 8, 4),      # as many codewords in four codebooks
    (1, 1025, True, 33, 31, 8, 4),     # the smallest summed in the L2; 1023 groups
    (1, 1025, False, 41, 25, 8, 0),
    (1, 2048, True, 41, 25, 8, 0),
    (1, 2048, False, 300, 129, 8, 4),
    (1, 2049, True, 33, 31, 8, 4),
    (2, 256, True, 1031, 33, 8, 4),    # several tiles per CTA, warps over two rows
    (2, 2, False, 3, 683, 8, 0),       # every group at two codewords; one group beyond two tiles
    (3, 250, True, 130, 64, 8, 0),
    (4, 256, False, 64, 70, 8, 4),
    (1, 2, True, 1, 1, 8, 0),          # one group
    (1, 300, True, 65, 17, 16, 4),     # groups of 16
]


def test_the_cases_are_on_both_sides_of_the_rule():
    source = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_14852_b200", "csrc", "pvt_pstep.cu")
    line = int(re.search(r"kPsSmallBins = (\d+);", open(source).read()).group(1))
    for f16 in (True, False):
        assert {line, line + 1} <= {M * K for M, K, cb, _, _, gd, _ in CASES if cb == f16 and gd == 8}


@pytest.mark.gpu
@pytest.mark.parametrize("M,K,f16,rows,per_row,gd,offset", CASES)
def test_gradients_at_the_edges(M, K, f16, rows, per_row, gd, offset):
    rng = np.random.default_rng(M * 1000 + K)
    cols, G = per_row * gd, rows * per_row
    g = rng.normal(0.0, 1e-3, size=(rows, cols)).astype(np.float32)
    scale = rng.uniform(0.5, 1.5, size=rows).astype(np.float32)
    books = rng.normal(size=(M, K, gd)).astype(np.float16 if f16 else np.float32)
    codes = rng.integers(0, K, size=(G, M)).astype(np.uint8 if K <= 256 else np.uint16)
    want_b, want_s = oracle.pstep_grad(g, scale, codes, books, rows, cols)
    flat = torch.empty(rows * cols + offset, dtype=torch.float32, device="cuda")
    view = flat[offset:].view(rows, cols)
    view.copy_(torch.from_numpy(g))
    up = lambda a: torch.from_numpy(a).cuda()
    scale_d, books_d, codes_d = up(scale), up(books), up(codes)
    desc = B.make_layer(rows, cols, None, view, scale_d, books_d, codes_d, group_dim=gd)
    gb = torch.full((M, K, gd), 7.0, dtype=torch.float64, device="cuda")
    gs = torch.full((rows,), 7.0, dtype=torch.float64, device="cuda")
    B.pvt_pstep_grad(desc, gb, gs)
    torch.cuda.synchronize()
    # n terms of magnitude <= a, added in another order
    assert np.abs(gb.cpu().numpy() - want_b).max() <= G * 1.5 * np.abs(g).max() * 2.0 ** -50
    assert np.abs(gs.cpu().numpy() - want_s).max() <= cols * np.abs(g).max() * np.abs(books.astype(np.float32)).max() * M * 2.0 ** -50


@pytest.mark.gpu
@pytest.mark.parametrize("n,offset", [(4, 0), (8, 0), (12, 0), (2052, 4), (303112, 0)])
def test_the_direction_may_take_the_place_of_the_gradient(n, offset):
    rng = np.random.default_rng(n)
    grad = rng.normal(0.0, 1e-3, size=n).astype(np.float32)
    m, v = rng.normal(0.0, 1e-3, size=n).astype(np.float32), rng.uniform(0.0, 1e-6, size=n).astype(np.float32)
    flat = [torch.zeros(n + offset, dtype=torch.float32, device="cuda")[offset:] for _ in range(3)]
    for t, a in zip(flat, (grad, m, v)):
        t.copy_(torch.from_numpy(a))
    want = oracle.adam_direction(grad, m, v, 3)
    B.pvt_adam_direction(flat[0], flat[1], flat[2], flat[0], 3)
    torch.cuda.synchronize()
    for t, a in zip(flat, (want, m, v)):
        assert t.cpu().numpy().tobytes() == a.tobytes()
