"""Row sorts of the orientation at the edges of their tiers: books (two adjacent hubs over d shared pages) with
scattered ids, whose triangles and 4-cycles are found by searching the hubs' rows; several books in one graph and in
a batch, hubs in graphs of one bitmap window, of several, and of too many ranks for bitmaps."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
C = math.comb
SIZES = (15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1022, 1023, 1024, 1025, 2047,
         2048, 2049, 4094, 4095, 4096, 4097, 9001)


@pytest.fixture(scope="module")
def harp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_12074_gb300 import _build, harp as H
    _build.build()
    H.lib()
    return H


def books(sizes, n, seed):
    """Disjoint books on random ids below n; [star3, path4, paw, cycle4, diamond, clique4] in closed form."""
    ids = np.random.RandomState(seed).permutation(n)[:sum(d + 2 for d in sizes)].astype(np.int32)
    src, dst, at = [], [], 0
    for d in sizes:
        a, b, pages = ids[at], ids[at + 1], ids[at + 2:at + 2 + d]
        at += d + 2
        src += [[a], np.full(d, a), np.full(d, b)]
        dst += [[b], pages, pages]
    want = [sum(2 * C(d, 3) for d in sizes), 0, 0, 0, sum(C(d, 2) for d in sizes), 0]
    return n, np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32), want


@pytest.mark.parametrize("d", SIZES)
def test_one_book(harp, d):
    n, s, t, want = books([d], d + 40, d)
    assert harp.count4_edges(n, s, t).tolist() == want


@pytest.mark.parametrize("n", [40_000, 1_605_632, 1_605_633, 2_000_001, 6_422_529], ids=lambda n: f"n{n}")
def test_books_by_ranks(harp, n):
    n, s, t, want = books(SIZES, n, 7)
    assert harp.count4_edges(n, s, t).tolist() == want


def test_books_in_a_batch(harp):
    members = [books([d], d + 40, d) for d in SIZES] + [books(SIZES, 50_000, 9)]
    hs = [harp.harp_build_csr(n, s, t) for n, s, t, _ in members]
    try:
        assert harp.harp_count4_batch(hs).tolist() == [w for *_, w in members]
    finally:
        for h in hs:
            h.close()
