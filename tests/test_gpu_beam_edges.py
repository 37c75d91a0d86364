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
