"""Parity of pvt_vstep_refine (local search over single-code changes, Appendix D) with the CPU checker.  Both
sides decide every move on the same binary64 errors under the same total order, so codes, move counts and
errors are compared exactly."""
import numpy as np
import pytest
import torch

import helpers
from oracle import pvt_oracle as oracle
from paper_2405_14852_b200 import binding as B
from paper_2405_14852_b200 import synth
from paper_2405_14852_b200.vstep import VStepLayer

pytestmark = pytest.mark.gpu


def oracle_nearest(X, C):
    return oracle.encode(X, C[None], np.zeros((X.shape[0], 1))).codes[:, 0]


def gpu_refine(L, idx_np, max_moves, encode_first=False):
    dev = VStepLayer.from_host(L)
    idx = torch.from_numpy(idx_np.astype(np.int32)).cuda()
    k = idx_np.size
    if encode_first:
        dev.encode(idx)
    err = torch.full((k,), -1.0, dtype=torch.float32, device="cuda")
    moves = torch.full((k,), 9999, dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.pvt_vstep_refine(dev.desc, idx, k, max_moves, err, moves, status)
    torch.cuda.synchronize()
    return dev.codes.cpu().numpy(), err.cpu().numpy(), moves.cpu().numpy(), int(status.item())


@pytest.mark.parametrize("M,K,f16,rows,cols,k", [
    (2, 256, True, 64, 512, 1500),
    (2, 200, False, 33, 72, 297),      # every group, ragged sizes
    (1, 256, False, 64, 256, 900),
    (3, 64, True, 64, 256, 600),
    (4, 256, True, 32, 512, 300),      # the largest codebooks in shared memory
    (4, 16, False, 32, 128, 512),
    (1, 2048, True, 64, 512, 333),     # two-byte codes; codebook read through L2 instead of shared memory
])
@pytest.mark.parametrize("max_moves", [0, 1, 64])
def test_refine_from_given_codes_matches_checker(M, K, f16, rows, cols, k, max_moves):
    L = synth.make_layer(rows, cols, cfg=200 + M, num_codebooks=M, codebook_size=K, codebook_fp16=f16,
                         nearest=oracle_nearest)  # stored codes are random: several moves per group
    G = L.num_groups
    idx = np.sort(np.random.default_rng(k).choice(G, size=k, replace=False)).astype(np.uint32)
    t = oracle.targets(L.W, L.g, L.scale, L.eta, idx)
    start = L.codes.reshape(G, M)[idx.astype(np.int64)]
    want, d, want_moves = oracle.local_search(t, L.codebooks, start, max_moves)
    codes, err, moves, status = gpu_refine(L, idx, max_moves)
    assert status == 0
    got = codes.reshape(G, M)
    assert np.array_equal(got[idx.astype(np.int64)].astype(np.int32), want)
    assert np.array_equal(moves, want_moves)
    assert np.array_equal(err, d.astype(np.float32))
    rest = np.setdiff1d(np.arange(G), idx.astype(np.int64))
    assert np.array_equal(got[rest], L.codes.reshape(G, M)[rest])
    if max_moves == 0:
        assert np.array_equal(got, L.codes.reshape(G, M))
    if M == 1 and max_moves >= 1:  # one move of a single codebook is the exhaustive search
        enc = oracle.encode(t, L.codebooks, start)
        assert np.array_equal(want, enc.codes)


def test_refine_after_the_beam_search_only_improves():
    L = synth.make_layer(96, 512, cfg=205, num_codebooks=2, codebook_size=256, codebook_fp16=True,
                         nearest=oracle_nearest, beam=1)  # greedy search: leaves improvable groups
    G = L.num_groups
    idx = oracle.select(oracle.group_norms(L.g, L.eta), 2000)
    t = oracle.targets(L.W, L.g, L.scale, L.eta, idx)
    enc = oracle.encode(t, L.codebooks, L.codes[idx.astype(np.int64)], L.beam)
    want, d, want_moves = oracle.local_search(t, L.codebooks, enc.codes)
    codes, err, moves, status = gpu_refine(L, idx, 64, encode_first=True)
    assert status == 0
    got = codes.reshape(G, 2)[idx.astype(np.int64)].astype(np.int32)
    decisive = (enc.d_second - enc.d_best) > 1e-6 * enc.d_second   # same start on both sides
    assert np.array_equal(got[decisive], want[decisive])
    assert np.array_equal(moves[decisive], want_moves[decisive])
    d_got = helpers.recon_error(t, L.codebooks, got)
    assert np.all(d_got <= enc.d_best * (1 + 1e-12))
    assert want_moves.sum() > 0, "the case should contain groups the beam search leaves improvable"


def test_refine_flags_bad_indices_and_codes():
    L = synth.make_layer(32, 128, cfg=206, num_codebooks=2, codebook_size=100, codebook_fp16=True,
                         nearest=oracle_nearest)
    L.codes[7, 1] = 100  # out of range
    idx = np.array([3, 7, 11, 5000], dtype=np.uint32)  # 5000 >= G = 512
    codes, err, moves, status = gpu_refine(L, idx, 8)
    assert status == (B.PVT_DEV_BAD_INDEX | B.PVT_DEV_BAD_CODE)
    assert np.array_equal(codes.reshape(-1, 2)[7], L.codes[7])


def test_refine_rejects_bad_arguments():
    L = synth.make_layer(32, 128, cfg=207, codebook_size=64, codebook_fp16=True)
    dev = VStepLayer.from_host(L)
    idx = torch.zeros(4, dtype=torch.int32, device="cuda")
    for k, mm in ((0, 1), (4, -1), (4, 70000), (10**6, 1)):
        with pytest.raises(B.PvtError) as e:
            B.pvt_vstep_refine(dev.desc, idx, k, mm)
        assert e.value.code == B.PVT_EINVAL


@pytest.mark.parametrize("M,K,f16,k", [
    (2, 100, True, 9473),    # one target in the last group of sixteen
    (3, 64, False, 5000),    # staged, two resident blocks per SM: more targets than twice the resident warps
    (1, 600, True, 19001),   # nothing staged: more than the doubled grid takes at once
    (4, 200, True, 9500),
])
def test_refine_with_more_targets_than_resident_warps(M, K, f16, k):
    L = synth.make_layer(320, 512, cfg=208, num_codebooks=M, codebook_size=K, codebook_fp16=f16, nearest=oracle_nearest)
    G = L.num_groups
    idx = np.sort(np.random.default_rng(k).choice(G, size=k, replace=False)).astype(np.uint32)
    at = idx.astype(np.int64)
    t = oracle.targets(L.W, L.g, L.scale, L.eta, idx)
    want, d, want_moves = oracle.local_search(t, L.codebooks, L.codes.reshape(G, M)[at], 2)
    codes, err, moves, status = gpu_refine(L, idx, 2)
    assert status == 0
    assert np.array_equal(codes.reshape(G, M)[at].astype(np.int32), want)
    assert np.array_equal(moves, want_moves) and np.array_equal(err, d.astype(np.float32))
    rest = np.setdiff1d(np.arange(G), at)
    assert np.array_equal(codes.reshape(G, M)[rest], L.codes.reshape(G, M)[rest])


@pytest.mark.parametrize("M,K,k,max_moves,start", [
    (2, 5, 1, 8, "random"),       # one target in a group of sixteen, codebooks smaller than a cell
    (2, 31, 17, 8, "random"),     # one target in the second group
    (3, 256, 33, 8, "search"),    # an odd codebook: half of the last pair of row tiles is empty
    (4, 255, 130, 8, "search"),
    (2, 33, 60001, 2, "mixed"),   # more groups than warps: several trips per block, some targets searched, some not
    (2, 64, 4000, 8, "equal"),    # every codeword twice: neighbours of the same error
    (2, 2, 40, 8, "random"),      # a pair of codewords per codebook
    (3, 17, 500, 16, "mixed"),    # one codeword in the second round of sixteen, and one beyond the codebook beside it
    (4, 16, 500, 16, "mixed"),
])
def test_refine_over_groups_of_targets(M, K, k, max_moves, start):
    rows, cols = (960, 512) if k > 5000 else (64, 512)
    L = synth.make_layer(rows, cols, cfg=209, num_codebooks=M, codebook_size=K, codebook_fp16=True, nearest=oracle_nearest)
    G = L.num_groups
    rng = np.random.default_rng(k)
    idx = np.sort(rng.choice(G, size=k, replace=False)).astype(np.uint32)
    at = idx.astype(np.int64)
    t = oracle.targets(L.W, L.g, L.scale, L.eta, idx)
    if start == "equal":
        L.codebooks[:, 1::2] = L.codebooks[:, 0::2]
    codes = L.codes.reshape(G, M)
    if start in ("search", "mixed"):
        found = oracle.encode(t, L.codebooks, codes[at], L.beam).codes
        codes[at] = np.where(rng.random((k, 1)) < (0.2 if start == "mixed" else 0.0), codes[at], found)
    want, d, want_moves = oracle.local_search(t, L.codebooks, codes[at], max_moves)
    got, err, moves, status = gpu_refine(L, idx, max_moves)
    assert status == 0
    assert np.array_equal(got.reshape(G, M)[at].astype(np.int32), want)
    assert np.array_equal(moves, want_moves) and np.array_equal(err, d.astype(np.float32))


def test_refine_beside_a_target_that_is_not_finite():
    L = synth.make_layer(64, 512, cfg=210, num_codebooks=2, codebook_size=100, codebook_fp16=True, nearest=oracle_nearest)
    idx = np.arange(0, 3000, 3, dtype=np.uint32)
    at = idx.astype(np.int64)
    t = oracle.targets(L.W, L.g, L.scale, L.eta, idx)
    want, d, want_moves = oracle.local_search(t, L.codebooks, L.codes[at], 8)
    L.W.reshape(-1, 8)[at[[5, 6, 700]], 3] = np.inf
    got, err, moves, status = gpu_refine(L, idx, 8)
    rest = np.setdiff1d(np.arange(1000), [5, 6, 700])
    assert np.array_equal(got.reshape(-1, 2)[at][rest].astype(np.int32), want[rest])
    assert np.array_equal(moves[rest], want_moves[rest]) and np.array_equal(err[rest], d.astype(np.float32)[rest])
    assert np.array_equal(got.reshape(-1, 2)[at][[5, 6, 700]], L.codes[at][[5, 6, 700]])


@pytest.mark.parametrize("M,K", [(2, 251), (3, 64), (4, 33)])
@pytest.mark.parametrize("size", [2.0 ** 20, 2.0 ** 60, 2.0 ** 66, 2.0 ** 117])
def test_refine_beside_targets_of_large_elements(M, K, size):
    """distances that binary32 cannot tell apart, or that leave its range: binary64 decides between all neighbours"""
    L = synth.make_layer(64, 512, cfg=211, num_codebooks=M, codebook_size=K, codebook_fp16=True, nearest=oracle_nearest)
    rng = np.random.default_rng(K)
    large = np.arange(1, L.num_groups, 16)
    L.W.reshape(-1, 8)[large] = rng.choice([-1.0, 1.0], (large.size, 8)) * size * L.scale[large // (L.cols // 8), None]
    idx = np.arange(L.num_groups, dtype=np.uint32)
    t = oracle.targets(L.W, L.g, L.scale, L.eta, idx)
    assert np.isfinite(t).all()
    want, d, want_moves = oracle.local_search(t, L.codebooks, L.codes.reshape(-1, M), 8)
    got, err, moves, status = gpu_refine(L, idx, 8)
    assert status == 0
    assert np.array_equal(got.reshape(-1, M).astype(np.int32), want)
    with np.errstate(over="ignore"):
        assert np.array_equal(moves, want_moves) and np.array_equal(err, d.astype(np.float32))
