"""The tensor search over codewords and targets in spatial order (many targets, a codebook of more than 32768 codewords)
against the FP32 engine, which tries every codeword of every target: codes and errors are the same to the bit."""
import pytest
import torch

import test_gpu_parity as parity
from paper_2405_14852_b200 import binding as B
from paper_2405_14852_b200.vstep import VStepLayer

pytestmark = pytest.mark.gpu


def enough(K):
    """targets from which on the order is worth its making"""
    return -(-3 * 10 ** 15 // (K * K))


def layer(rows, cols, K, seed, change=None):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    W = torch.randn(rows, cols, generator=gen, device="cuda").mul_(0.02)
    g = torch.randn(rows, cols, generator=gen, device="cuda").mul_(1e-3)
    scale = W.abs().amax(1)
    G = W.numel() // 8
    pick = torch.randperm(G, generator=gen, device="cuda")[:K]
    books = (W.view(-1, 8)[pick] / scale[pick // (cols // 8), None]).half()[None].contiguous()
    codes = torch.randint(0, K, (G, 1), generator=gen, device="cuda").to(torch.int16)
    if change:
        change(W, g, scale, books[0], codes)
    return W, g, scale, books, codes


def check(parts, idx, again=False, other="fp32", fill=None):
    """other: the engine to compare with, on the targets in portions too small for the order; fill: what every 16 bits of the
    workspace behind its header hold before the call"""
    W, g, scale, books, codes = parts
    rows, cols = W.shape
    got = []
    for engine, portion in (("tensor", idx.numel()), (other, enough(65536) // 2)):
        own = codes.clone()
        err = torch.full((idx.numel(),), -1.0, device="cuda")
        with parity.search_engine(engine):
            L = VStepLayer(rows, cols, W, g, scale, books, own, max_k=portion)
            if fill is not None:
                L.reserve(portion)[256:].view(torch.int16).fill_(fill)
            for _ in range(1 + again):
                for at in range(0, idx.numel(), portion):
                    L.encode(idx[at:at + portion].contiguous(), err[at:at + portion])
            torch.cuda.synchronize()
            assert L.status() == 0
        got.append((own, err))
    assert torch.equal(got[0][0], got[1][0])
    assert torch.equal(got[0][1], got[1][1])
    # without errors to report, a codeword that binary32 tells from all others is taken as it is
    own = codes.clone()
    L = VStepLayer(rows, cols, W, g, scale, books, own, max_k=idx.numel())
    for _ in range(1 + again):
        L.encode(idx)
    torch.cuda.synchronize()
    assert L.status() == 0
    assert torch.equal(own, got[0][0])


@pytest.mark.parametrize("K,more", [
    (65536, 0), (65536, 513), (65535, 300001), (50048, 1), (40000, 255),  # a last step that is full, and one that is not
    (32769, 77),  # the smallest: the last step has one codeword
])
def test_same_codes_as_the_exhaustive_search(K, more):
    k = enough(K) + more
    parts = layer(4096, 8192, K, K + k)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(k)
    idx = torch.randperm(4096 * 1024, generator=gen, device="cuda")[:k].int()
    check(parts, idx)
    check(parts, idx.sort().values, again=True)  # from stored codes that are the nearest


def equal_codewords(W, g, scale, book, codes):
    book[1000:30000] = book[31000:60000]


def few_values(W, g, scale, book, codes):
    book.copy_((book * 4).round() / 4)  # most codewords many times over


def one_dimension(W, g, scale, book, codes):
    book[:, 1:] = 0


def timed(parts, idx):
    """least time of a search over the lists, one after the other, and the codes that it leaves"""
    W, g, scale, books, codes = parts
    own = codes.clone()
    L = VStepLayer(*W.shape, W, g, scale, books, own, max_k=max(i.numel() for i in idx))
    idx = [i.contiguous() for i in idx]
    took = []
    for _ in range(4):
        start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        start.record()
        for i in idx:
            L.encode(i)
        end.record()
        torch.cuda.synchronize()
        took.append(start.elapsed_time(end))
    return min(took), own


def one_codeword(W, g, scale, book, codes):
    book.copy_(book[:1].expand_as(book))


def outliers(W, g, scale, book, codes):
    book[::97] *= 400.0     # beyond the scaled range of most boxes
    book[5::5003] = 300.0   # not in the operand image
    book[7::9001] = -60000.0
    book[11, 3] = float("inf")
    book[13, 2] = float("nan")
    book[17, 2] = float("-inf")
    book[19] = -book[13]


def far_targets(W, g, scale, book, codes):
    scale[3] = 1e-4    # elements up to 256 and beyond
    scale[4] = 1e-3
    scale[5] = 1e6     # next to zero
    scale[6] *= 0.1


def small_codewords(W, g, scale, book, codes):
    book.mul_(2.0 ** -10)


def large_codewords(W, g, scale, book, codes):
    book.mul_(64.0)


def bad_codes(W, g, scale, book, codes):
    codes.fill_(-1)  # stored codes beyond the codebook: no bound to begin with


def spread_dimensions(W, g, scale, book, codes):
    f = torch.tensor([1, 0.5, 0.25, 0.1, 4, 0.01, 1, 2], device="cuda")
    W.view(-1, 8).mul_(f)
    g.view(-1, 8).mul_(f)
    book.mul_(f.half())


@pytest.mark.parametrize("change", [equal_codewords, few_values, one_dimension, one_codeword, outliers, far_targets,
                                    small_codewords, large_codewords, bad_codes, spread_dimensions])
def test_unusual_inputs(change):
    K = 60000
    parts = layer(4096, 2048, K, 7, change)
    idx = torch.arange(enough(K), dtype=torch.int32, device="cuda")
    check(parts, idx, other="tensor")  # (which takes codewords that are no numbers)


def repeated_codewords(W, g, scale, book, codes):
    book[256:] = book[:256].repeat(-(-book.shape[0] // 256), 1)[256:book.shape[0]]


def dead_codewords(W, g, scale, book, codes):
    book.abs_()
    book[torch.arange(book.shape[0], device="cuda") % 50 < 27] = 0


@pytest.mark.parametrize("fill", [5, 300])  # numbers of steps that exist
@pytest.mark.parametrize("K", [60000, 65536])
@pytest.mark.parametrize("change", [one_codeword, repeated_codewords, dead_codewords])
def test_equal_codewords_whatever_the_workspace_holds(change, K, fill):
    """Steps whose boxes have the same centre: every place of the list of near ones is written (test_sorted_near_steps.py)."""
    parts = layer(4096, 2048, K, 8, change)
    idx = torch.arange(enough(K), dtype=torch.int32, device="cuda")
    check(parts, idx, other="tensor", fill=fill)


def unlike_groups(W, g, scale, book, codes):
    """groups of unlike size: beside the largest of a row most are next to zero, and so are most codewords"""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(2)
    W.view(-1, 8).mul_(torch.exp(torch.randn(codes.shape[0], 1, generator=gen, device="cuda")))
    scale.copy_(W.abs().amax(1))
    pick = torch.randperm(codes.shape[0], generator=gen, device="cuda")[:book.shape[0]]
    book.copy_((W.view(-1, 8)[pick] / scale[pick // (W.shape[1] // 8), None]).half())


@pytest.mark.parametrize("change", [one_codeword, unlike_groups])
def test_codewords_too_many_to_remember_are_gone_over_once(change):
    """Where more codewords are near than a record holds, all that it stands for are evaluated, and none twice: the search in
    spatial order takes no longer than the one of every codeword (1.7 times as long when it visited all for each record)."""
    K = 60000
    parts = layer(4096, 2048, K, 9, change)
    every = torch.arange(enough(K), dtype=torch.int32, device="cuda")
    whole, portions = timed(parts, [every]), timed(parts, every.chunk(2))
    assert torch.equal(whole[1], portions[1])
    assert whole[0] < 1.25 * portions[0]


def pruned(W, g, scale, book, codes):
    zero = torch.arange(codes.shape[0], device="cuda") % 10 != 0
    W.view(-1, 8)[zero] = 0
    g.view(-1, 8)[zero] = 0


def test_many_equal_targets_do_not_queue():
    """Nine of ten groups are zero: they all fall into one cell of the tree.  (Counted one by one they took 1.6 times as long as
    targets that are spread.)"""
    idx = torch.arange(4096 * 1024, dtype=torch.int32, device="cuda")
    spread, equal = [timed(layer(4096, 8192, 65536, 10, change), [idx])[0] for change in (None, pruned)]
    assert equal < 1.25 * spread


def test_the_search_counts_what_it_evaluates():
    W, g, scale, books, codes = layer(4096, 2048, 65536, 11)
    k = enough(65536) + 100
    L = VStepLayer(4096, 2048, W, g, scale, books, codes, max_k=k)
    L.encode(torch.arange(k, dtype=torch.int32, device="cuda"))
    assert 0.4 < B.pvt_evaluated_share(L.desc, k, L.reserve(k)) < 0.7  # normally distributed weights
    assert B.pvt_evaluated_share(L.desc, enough(65536) // 2, L.reserve(k)) == 1.0
    books[0].copy_(books[0][:1].expand_as(books[0]))
    L.encode(torch.arange(k, dtype=torch.int32, device="cuda"))
    assert B.pvt_evaluated_share(L.desc, k, L.reserve(k)) == 1.0  # equal codewords: all of them


def test_an_index_out_of_range_is_reported():
    W, g, scale, books, codes = layer(4096, 2048, 65536, 3)
    idx = torch.arange(enough(65536), dtype=torch.int32, device="cuda")
    idx[12345] = 4096 * 256
    L = VStepLayer(4096, 2048, W, g, scale, books, codes, max_k=idx.numel())
    L.encode(idx)
    torch.cuda.synchronize()
    assert L.status() == 1


@pytest.mark.parametrize("withhold", [0, 11])
def test_a_wait_that_runs_out_is_reported_and_the_next_call_is_correct(withhold):
    """The bounded waits (test_gpu_wait_limit.py) where a unit is a tile and a copy a step of its list."""
    K = 65536
    W, g, scale, books, codes = layer(4096, 2048, K, 4)
    idx = torch.arange(enough(K), dtype=torch.int32, device="cuda")
    own = codes.clone()
    L = VStepLayer(4096, 2048, W, g, scale, books, own, max_k=idx.numel())
    B.pvt_test_wait_limit(20000, withhold)
    try:
        L.encode(idx)
        torch.cuda.synchronize()
        status = L.status()
    finally:
        B.pvt_test_wait_limit(0, -1)
    assert status & B.PVT_DEV_WAIT_EXPIRED
    own.copy_(codes)
    L.encode(idx)
    torch.cuda.synchronize()
    assert L.status() == 0
    other = codes.clone()
    portion = enough(K) // 2
    M = VStepLayer(4096, 2048, W, g, scale, books, other, max_k=portion)
    for at in range(0, idx.numel(), portion):
        M.encode(idx[at:at + portion].contiguous())
    torch.cuda.synchronize()
    assert torch.equal(own, other)
