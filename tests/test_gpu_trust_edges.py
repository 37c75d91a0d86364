"""Trust-ratio step where the ranking sort and the summed changes change shape: one block, another round of pairs per
thread, the last size that is sorted in one kernel per digit and the first beyond; norms with many ties."""
import numpy as np
import pytest

from paper_2405_14852_b200 import synth
from test_gpu_trust import run_case, settle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k_max,ratio", [
    (1, 0.05), (255, 0.02), (257, 0.02), (16384, 0.03), (16385, 0.03), (131073, 0.05), (524288, 0.05), (524289, 0.2),
])
def test_trust_step_at_the_sort_edges(k_max, ratio):
    rows, cols = (2048, 2080) if k_max > 20000 else (512, 272)
    L = settle(synth.make_layer(rows, cols, cfg=197, codebook_size=16, codebook_fp16=False))
    L.g = np.round(L.g, 3)  # few distinct values: equal norms
    run_case(L, k_max, ratio)


@pytest.mark.parametrize("rows,cols,k_max", [
    (16, 264, 100),        # one trip of the norm: three of its four shares are empty
    (2048, 2400, 3000),    # two trips
    (4096, 6080, 3000),    # six: shares of one and two
])
def test_trust_step_with_uneven_shares_of_the_norm(rows, cols, k_max):
    run_case(settle(synth.make_layer(rows, cols, cfg=198, codebook_size=16, codebook_fp16=True)), k_max, 0.02)
