"""Selection at the sizes where its passes change: groups that do not fill a word of 32, update matrices on a 16-byte
but not a 32-byte boundary, one and several trips per CTA, a threshold bin that holds nearly everything."""
import numpy as np
import pytest
import torch

from oracle import pvt_oracle as oracle
from paper_2405_14852_b200 import binding as B


@pytest.mark.gpu
@pytest.mark.parametrize("rows,cols,k,offset,levels", [
    (1, 8, 1, 0, 0),            # one group
    (3, 88, 32, 4, 0),          # 33 groups, one bit in the second word, unaligned
    (257, 264, 8000, 4, 0),     # unaligned, odd groups per row
    (513, 1032, 66176, 0, 0),   # all but one group
    (4099, 136, 17, 0, 3),      # three norms only: ties in every word
    (20003, 2008, 51234, 0, 0),  # more than 32768 groups per CTA: several trips
    (20003, 2008, 2500000, 4, 2),
])
def test_selection_edges(rows, cols, k, offset, levels):
    rng = np.random.default_rng(rows * 7 + k)
    g = rng.normal(0.0, 1e-3, size=(rows, cols)).astype(np.float32)
    if levels:
        g = np.repeat(rng.integers(1, levels + 1, size=(rows, cols // 8)), 8, axis=1).astype(np.float32) * np.float32(1e-3)
    want = oracle.select(oracle.group_norms(g, 1.0), k)
    flat = torch.empty(rows * cols + offset, dtype=torch.float32, device="cuda")
    view = flat[offset:].view(rows, cols)
    view.copy_(torch.from_numpy(g))
    desc = B.pvt_layer(rows, cols, 8, 1, 256, B.PVT_F16, B.PVT_U8, 8, 1.0, 0, None, view.data_ptr(), None, None, None)
    ws = B.new_workspace(desc, k)
    idx = torch.full((k,), -1, dtype=torch.int32, device="cuda")
    for _ in range(2):  # the second call finds the workspace as the first left it
        B.pvt_vstep_select(desc, k, idx, ws)
    assert B.pvt_status(ws) == 0
    assert np.array_equal(idx.cpu().numpy().astype(np.uint32), np.asarray(want, dtype=np.uint32))


@pytest.mark.gpu
@pytest.mark.parametrize("rows,cols,k,offset,levels", [
    (4096, 9184, 47001, 0, 0),     # 148 CTAs of 993 words: the first size with more CTAs than SMs in the last pass
    (16003, 2440, 48809, 0, 0),    # more words than threads per SM: two CTAs of an SM
    (16003, 2440, 1000000, 0, 2),  # the same with ties in every word
    (20003, 3928, 98214, 0, 0),    # and several trips of those
    (1031, 32, 900, 0, 1),         # one norm only
])
def test_selection_edges_of_the_last_pass(rows, cols, k, offset, levels):
    test_selection_edges(rows, cols, k, offset, levels)
