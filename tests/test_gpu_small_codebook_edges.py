"""Search over one small codebook at the edges of its kernel: blocks of 16 codewords, the largest codebook, tiles of 32
and 64 targets, both splits of the targets."""
import numpy as np
import pytest

from paper_2405_14852_b200 import synth
from test_gpu_parity import check_encode

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,f16,k", [
    (2, False, 1), (15, True, 31), (16, False, 32), (17, True, 33), (255, False, 64), (256, True, 65),
    (1000, True, 37887), (1023, False, 37888), (1024, True, 37889), (300, False, 40000),
])
def test_small_codebook_search_at_its_edges(K, f16, k):
    rows, cols = (128, 64) if k < 1000 else (640, 512)
    L = synth.make_layer(rows, cols, cfg=210, codebook_size=K, codebook_fp16=f16)
    idx = np.sort(np.random.default_rng(k).permutation(L.num_groups)[:k]).astype(np.uint32)
    check_encode(L, idx)
