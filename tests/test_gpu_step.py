"""A step as one call against its three calls: few groups of many (all weights are dequantised beside the selection and those
of the chosen groups again after the search), on both sides of that rule, over every representation."""
import pytest
import torch

from paper_2405_14852_b200.vstep import VStepLayer

pytestmark = pytest.mark.gpu

CASES = [  # rows, cols, codebooks, codewords, group, codebook type, codes, k
    (64, 72, 1, 200, 8, torch.float16, torch.uint8, 72),          # more than are dequantised first
    (64, 72, 1, 200, 8, torch.float32, torch.uint8, 73),          # (fp32 codebooks, fp16 weights: one above an eighth)
    (64, 72, 1, 200, 8, torch.float32, torch.uint8, 72),          # (the most)
    (64, 72, 1, 200, 8, torch.float16, torch.uint8, 36),          # the most of the others: a sixteenth; one more
    (64, 72, 1, 200, 8, torch.float16, torch.uint8, 37),
    (1000, 2008, 3, 256, 8, torch.float16, torch.uint8, 1000),    # three and four codebooks with enough groups
    (1000, 2008, 4, 256, 8, torch.float32, torch.uint8, 3921),    # a 64th
    (16384, 4096, 1, 100, 8, torch.float16, torch.uint8, 300000),  # the most groups of a small codebook, and one more
    (16384, 4096, 1, 100, 8, torch.float16, torch.uint8, 300001),
    (11264, 8192, 1, 65536, 8, torch.float16, torch.int16, 700000),  # a search in spatial order
    (3, 8, 1, 2, 8, torch.float16, torch.uint8, 1),
    (16, 8, 1, 2, 8, torch.float16, torch.uint8, 2),              # fewer groups than threads of a block
    (300, 1000, 1, 5000, 8, torch.float16, torch.int16, 1000),
    (2048, 2048, 1, 60000, 8, torch.float16, torch.int16, 5003),  # every block has several trips
    (257, 1032, 1, 1000, 8, torch.float32, torch.int16, 3000),
    (257, 1032, 1, 2000, 8, torch.float32, torch.int16, 3000),
    (129, 264, 2, 256, 8, torch.float16, torch.uint8, 400),
    (129, 264, 2, 100, 8, torch.float32, torch.uint8, 400),
    (1000, 1000, 3, 256, 8, torch.float16, torch.uint8, 1000),
    (1000, 1000, 3, 31, 8, torch.float32, torch.uint8, 1000),
    (500, 1600, 4, 256, 8, torch.float16, torch.uint8, 777),      # three and four codebooks: too few groups
    (500, 520, 4, 256, 8, torch.float32, torch.uint8, 777),
    (1000, 1000, 4, 256, 8, torch.float32, torch.uint8, 777),
    (129, 272, 1, 1500, 16, torch.float16, torch.int16, 200),
    (129, 272, 1, 100, 16, torch.float32, torch.uint8, 200),
]


@pytest.mark.parametrize("out", [torch.float32, torch.float16])
@pytest.mark.parametrize("rows,cols,M,K,gd,book,code,k", CASES)
def test_a_step_is_its_three_calls(rows, cols, M, K, gd, book, code, k, out):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(rows + cols + M)
    W = torch.randn(rows, cols, generator=gen, device="cuda") * 0.02
    g = torch.randn(rows, cols, generator=gen, device="cuda") * 1e-3
    books = (torch.randn(M, K, gd, generator=gen, device="cuda") * 0.25).to(book)
    G = rows * cols // gd
    codes = torch.randint(0, K, (G, M), generator=gen, device="cuda").to(code)
    if K < 200:
        codes[G // 2] = -1 if code == torch.int16 else 255  # beyond the codebook: taken as the first codeword
    scale = W.abs().amax(1)
    got = []
    for whole in (True, False):
        own = codes.clone()
        L = VStepLayer(rows, cols, W, g, scale, books, own, max_k=k, group_dim=gd)
        W_hat = torch.full((rows, cols), 7.0, dtype=out, device="cuda")
        idx = torch.full((k,), -1, dtype=torch.int32, device="cuda")
        if whole:
            L.step(k, idx, W_hat)
        else:
            L.select(k, idx)
            L.encode(idx)
            L.dequant(W_hat)
        torch.cuda.synchronize()
        got.append((idx, own, W_hat, L.status()))
    assert all(torch.equal(a, b) for a, b in zip(got[0][:3], got[1][:3]))
    assert got[0][3] == got[1][3]


@pytest.mark.parametrize("what", ["W", "g"])
def test_weights_that_take_the_place_of_an_input(what):
    rows, cols, K, k = 128, 512, 300, 100
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    got = []
    W0 = torch.randn(rows, cols, generator=gen, device="cuda") * 0.02
    g0 = torch.randn(rows, cols, generator=gen, device="cuda") * 1e-3
    books = (torch.randn(1, K, 8, generator=gen, device="cuda") * 0.25).half()
    codes = torch.randint(0, K, (rows * cols // 8, 1), generator=gen, device="cuda").to(torch.int16)
    for whole in (True, False):
        W, g, own = W0.clone(), g0.clone(), codes.clone()
        L = VStepLayer(rows, cols, W, g, W0.abs().amax(1), books, own, max_k=k)
        W_hat = {"W": W, "g": g}[what]
        idx = torch.empty(k, dtype=torch.int32, device="cuda")
        if whole:
            L.step(k, idx, W_hat)
        else:
            L.select(k, idx)
            L.encode(idx)
            L.dequant(W_hat)
        torch.cuda.synchronize()
        got.append((idx, own, W_hat))
    assert all(torch.equal(a, b) for a, b in zip(*got))
