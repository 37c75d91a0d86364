"""Beam search over three and four codebooks where a middle stage's short list changes its way: codebooks of a few
codewords (fewer cells than kept tuples), sizes around 32, lists that overflow because codewords nearly coincide, and
because they do."""
import numpy as np
import pytest

from oracle import pvt_oracle as oracle
from paper_2405_14852_b200 import binding as B
from paper_2405_14852_b200 import synth
from test_gpu_parity import check_encode, oracle_nearest, run_encode


@pytest.mark.gpu
@pytest.mark.parametrize("M", [3, 4])
@pytest.mark.parametrize("K,beam,f16", [
    (2, 8, True), (3, 3, False), (7, 8, True), (8, 8, False), (9, 8, True), (31, 7, True), (33, 8, False), (255, 2, True),
])
def test_small_and_ragged_codebooks(M, K, beam, f16):
    L = synth.make_layer(16, 264, cfg=300 + M, num_codebooks=M, codebook_size=K, codebook_fp16=f16, beam=beam,
                         nearest=oracle_nearest)
    check_encode(L, np.arange(3, L.num_groups, 2, dtype=np.uint32))


@pytest.mark.gpu
@pytest.mark.parametrize("M", [3, 4])
@pytest.mark.parametrize("copies,jitter,f16", [(16, 1e-3, True), (16, 0.0, True), (32, 1e-6, False), (5, 0.0, False)])
def test_clustered_codewords(M, copies, jitter, f16):
    L = synth.make_layer(16, 256, cfg=310 + M, num_codebooks=M, codebook_size=256, codebook_fp16=f16,
                         nearest=oracle_nearest)
    rng = np.random.default_rng(copies)
    for m in range(1, M):
        base = L.codebooks[m].astype(np.float32)[np.arange(256) // copies]
        L.codebooks[m] = (base + rng.normal(0.0, jitter, size=base.shape)).astype(L.codebooks.dtype)
    check_encode(L, np.arange(L.num_groups, dtype=np.uint32))


@pytest.mark.gpu
@pytest.mark.parametrize("M,f16,value", [(2, True, np.nan), (2, False, np.nan), (2, True, np.inf), (3, True, np.nan)])
def test_a_target_that_is_not_finite_is_reported_and_keeps_its_codes(M, f16, value):
    L = synth.make_layer(16, 256, cfg=320 + M, num_codebooks=M, codebook_size=100, codebook_fp16=f16, nearest=oracle_nearest)
    odd = [2, 3, 77, L.num_groups - 1]  # two of one group of four targets, alone among others, the last
    idx = np.arange(L.num_groups, dtype=np.uint32)
    t = oracle.targets(L.W, L.g, L.scale, L.eta, idx)
    before = L.codes.reshape(-1, M).copy()
    want = oracle.encode(t, L.codebooks, before, L.beam)
    L.W.reshape(-1, 8)[odd, 5] = value
    got, _, status = run_encode(L, idx)
    assert status == B.PVT_DEV_INTERNAL
    got = got.reshape(-1, M)
    assert np.array_equal(got[odd], before[odd])
    rest = np.setdiff1d(idx, odd)
    decisive = (want.d_second - want.d_best)[rest] > 1e-6 * want.d_second[rest]
    assert np.array_equal(got[rest][decisive], want.codes[rest][decisive])


@pytest.mark.gpu
@pytest.mark.parametrize("M,K,beam,f16", [
    (2, 2, 8, True), (2, 3, 8, True), (2, 8, 8, True), (2, 9, 8, True), (2, 33, 8, True), (2, 251, 5, True), (2, 256, 1, True),
    (2, 9, 8, False), (2, 251, 5, False),
])
def test_small_and_ragged_first_codebook(M, K, beam, f16):
    L = synth.make_layer(16, 264, cfg=330 + M, num_codebooks=M, codebook_size=K, codebook_fp16=f16, beam=beam,
                         nearest=oracle_nearest)
    check_encode(L, np.arange(2, L.num_groups, 3, dtype=np.uint32))


@pytest.mark.gpu
@pytest.mark.parametrize("M", [2, 3])
@pytest.mark.parametrize("copies,jitter", [(16, 1e-3), (40, 1e-3), (16, 0.0), (40, 0.0), (32, 1e-6), (5, 0.0)])
def test_clustered_first_codebook(M, copies, jitter):
    """more codewords at the limit of stage 1 than its list holds, apart, nearly equal and equal"""
    L = synth.make_layer(16, 256, cfg=340 + M, num_codebooks=M, codebook_size=256, codebook_fp16=True, nearest=oracle_nearest)
    rng = np.random.default_rng(copies)
    base = L.codebooks[0].astype(np.float32)[np.arange(256) // copies]
    L.codebooks[0] = (base + rng.normal(0.0, jitter, size=base.shape)).astype(L.codebooks.dtype)
    check_encode(L, np.arange(L.num_groups, dtype=np.uint32))


@pytest.mark.gpu
@pytest.mark.parametrize("M", [2, 3, 4])
@pytest.mark.parametrize("K,size,f16", [
    (251, 2.0 ** 60, True), (251, 2.0 ** 66, True), (251, 2.0 ** 101, True), (251, 2.0 ** 117, True), (251, 2.0 ** 126.5, True),
    (251, 2.0 ** 127.9, True), (20, 2.0 ** 117, True), (251, 2.0 ** 60, False), (251, 2.0 ** 117, False),
])
def test_a_target_of_large_elements_beside_ordinary_ones(M, K, size, f16):
    """Scores of such a target are not to be told apart in binary32, or not finite; its distances are finite in binary64 and
    the same for all tuples (the elements of codewords are below half a unit of its own): the lowest tuple.  Half of the
    large targets have no valid previous tuple, so that nothing stands in for what the search finds."""
    L = synth.make_layer(16, 256, cfg=350 + M, num_codebooks=M, codebook_size=K, codebook_fp16=f16, nearest=oracle_nearest)
    large = np.arange(1, L.num_groups, 16)  # one of four targets, the others of its group of sixteen as they were
    rng = np.random.default_rng(M)
    elements = rng.choice([-1.0, 1.0], (large.size, 8)) * size * rng.uniform(0.5, 1.0, (large.size, 8))
    L.W.reshape(-1, 8)[large] = elements * L.scale[large // (L.cols // 8), None]
    idx = np.arange(L.num_groups, dtype=np.uint32)
    t = oracle.targets(L.W, L.g, L.scale, L.eta, idx)
    assert np.isfinite(t).all() and np.abs(t).max() > 0.5 * size
    codes = L.codes.reshape(-1, M)
    want = oracle.encode(t, L.codebooks, codes, L.beam)
    assert not want.codes[large].any()
    codes[large[::2], M - 1] = 255
    got, _, status = run_encode(L, idx)
    got = got.reshape(-1, M)
    assert status == B.PVT_DEV_BAD_CODE  # reported for the places that hold no code
    assert got.max() < K
    assert not got[large].any()
    rest = np.setdiff1d(idx, large)
    decisive = (want.d_second - want.d_best)[rest] > 1e-6 * want.d_second[rest]
    assert np.array_equal(got[rest][decisive], want.codes[rest][decisive])


@pytest.mark.gpu
@pytest.mark.parametrize("M,K", [(2, 256), (3, 251), (4, 64)])
@pytest.mark.parametrize("f16", [True, False])
def test_targets_of_very_different_sizes_side_by_side(M, K, f16):
    """the scores of a target owe nothing to the size of the other three of its group"""
    L = synth.make_layer(16, 264, cfg=360 + M, num_codebooks=M, codebook_size=K, codebook_fp16=f16, nearest=oracle_nearest)
    L.W.reshape(-1, 8)[:] *= np.exp2(np.random.default_rng(K).integers(-12, 13, (L.num_groups, 1))).astype(np.float32)
    check_encode(L, np.arange(L.num_groups, dtype=np.uint32))
