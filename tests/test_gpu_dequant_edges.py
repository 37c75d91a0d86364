"""Dequantisation where a thread makes several trips: the codes and scales of the next trip are asked for before the
results of this one are stored.  Results beyond one trip of all resident blocks, a last trip that is not full, one group
beyond it, a bad code in the last trip."""
import numpy as np
import pytest
import torch

from oracle import pvt_oracle as oracle
from paper_2405_14852_b200 import binding as B


@pytest.mark.gpu
@pytest.mark.parametrize("M,K,f16,gd,out_f16,rows,per_row", [
    (1, 300, True, 8, False, 1237, 1031),
    (1, 5000, True, 8, True, 1237, 1031),    # two-byte codes, codebook not staged
    (2, 256, False, 8, False, 401, 3203),
    (3, 77, True, 8, True, 1021, 1301),
    (4, 256, True, 8, False, 4099, 257),
    (1, 2000, True, 16, True, 601, 1511),
])
def test_dequant_over_several_trips(M, K, f16, gd, out_f16, rows, per_row):
    rng = np.random.default_rng(K)
    cols, G = per_row * gd, rows * per_row
    books = rng.normal(size=(M, K, gd)).astype(np.float16 if f16 else np.float32)
    scale = rng.uniform(0.5, 1.5, size=rows).astype(np.float32)
    codes = rng.integers(0, K, size=(G, M)).astype(np.uint8 if K <= 256 else np.uint16)
    want = oracle.dequant(codes, books, scale, rows, cols)
    up = lambda a: torch.from_numpy(a).cuda()
    scale_d, books_d, codes_d = up(scale), up(books), up(codes)
    desc = B.make_layer(rows, cols, None, None, scale_d, books_d, codes_d, group_dim=gd)
    out = torch.full((rows, cols), -7.0, dtype=torch.float16 if out_f16 else torch.float32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.pvt_dequant(desc, out, status)
    torch.cuda.synchronize()
    want = want.astype(np.float16) if out_f16 else want
    assert out.cpu().numpy().tobytes() == want.tobytes() and int(status.item()) == 0
    if K < 256 or K > 256:  # a code that is out of range, in the last group
        codes[-1, M - 1] = K
        codes_d.copy_(up(codes))
        B.pvt_dequant(desc, out, status)
        torch.cuda.synchronize()
        assert int(status.item()) == B.PVT_DEV_BAD_CODE
        assert out.cpu().numpy()[:-1].tobytes() == want[:-1].tobytes()
