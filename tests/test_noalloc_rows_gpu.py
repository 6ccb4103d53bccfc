"""harp_count4_noalloc on a caller's CSR that is not simple: repeats in hub rows (longer than the block sort takes)
are kept, as in shorter rows, so every array holds as many entries as the degrees say; rows that are not symmetric are
refused where more than m of their entries point upwards in rank, the most that the arrays have room for."""
from math import comb

import numpy as np
import pytest

import graphgen
import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def harp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_12074_gb300 import _build, harp as H
    _build.build()
    H.lib()
    return H


def csr_of(n, src, dst):
    """Offsets and columns of the arcs as given, repeats included, rows ascending."""
    key = np.sort(np.asarray(src, np.int64) * n + np.asarray(dst, np.int64))
    off = np.concatenate([[0], np.cumsum(np.bincount(key // n, minlength=n))])
    return off.astype(np.int64), (key % n).astype(np.int32)


def count(harp, n, off, cols):
    out = torch.full((16,), -1, dtype=torch.int64, device="cuda")
    o, c = torch.from_numpy(off).cuda(), torch.from_numpy(cols).cuda()
    harp.harp_count4_noalloc(n, cols.size // 2, o.data_ptr(), c.data_ptr(), out.data_ptr())
    torch.cuda.synchronize()
    return out.cpu().tolist()


def counts_normally(harp):
    g = graphgen.ba(6000, 4, 2)
    s, d = np.concatenate([g.src, g.dst]), np.concatenate([g.dst, g.src])
    off, cols = csr_of(g.n, s, d)
    out = count(harp, g.n, off, cols)
    assert out[:6] == O.count4_combo(g.n, g.src, g.dst).tolist() and out[6] == 0


def stars_with_repeated_edge(a, b, times):
    """Vertex 0 with a leaves and vertex 1 with b, joined by an edge that is listed several times."""
    n = 2 + a + b
    hub = np.concatenate([np.zeros(a, np.int64), np.ones(b, np.int64), np.zeros(times, np.int64)])
    other = np.concatenate([np.arange(2, n), np.ones(times, np.int64)])
    return n, np.concatenate([hub, other]), np.concatenate([other, hub])


@pytest.mark.parametrize("a,b,times", [(4094, 4200, 3), (5000, 6000, 3), (5000, 9000, 700)])
def test_repeats_in_hub_rows(harp, a, b, times):
    n, s, d = stars_with_repeated_edge(a, b, times)
    da, db = a + times, b + times
    out = count(harp, n, *csr_of(n, s, d))
    # stars at both hubs; paths of three edges through each copy of the middle edge
    assert out[:7] == [comb(da, 3) + comb(db, 3), times * (da - 1) * (db - 1), 0, 0, 0, 0, 0]
    counts_normally(harp)


def test_repeated_leaf_of_a_hub(harp):
    n = 5002  # one vertex isolated
    leaves = np.concatenate([np.arange(1, 5001), [5000]])
    hub = np.zeros(leaves.size, np.int64)
    out = count(harp, n, *csr_of(n, np.concatenate([hub, leaves]), np.concatenate([leaves, hub])))
    assert out[:7] == [comb(5001, 3), 2 * 5000, 0, 0, 0, 0, 0]
    counts_normally(harp)


def one_sided(k, heads):
    """k vertices list vertex 0, which lists others instead, so many that they sort below it."""
    n = 1 + k + heads
    src = np.concatenate([np.arange(1, k + 1), np.zeros(heads, np.int64)])
    dst = np.concatenate([np.zeros(k, np.int64), np.arange(k + 1, n)])
    return n, src, dst


@pytest.mark.parametrize("k,heads", [(4, 2), (1000, 2), (20_002, 20_000), (200_000, 40)])
def test_more_upward_entries_than_edges(harp, k, heads):
    n, s, d = one_sided(k, heads)
    out = count(harp, n, *csr_of(n, s, d))
    assert out[:6] == [0] * 6 and out[6] != 0
    counts_normally(harp)


@pytest.mark.parametrize("k,heads", [(0, 6), (20, 20), (1000, 9000)])
def test_other_one_sided_rows_pass(harp, k, heads):
    n, s, d = one_sided(k, heads)
    out = count(harp, n, *csr_of(n, s, d))
    assert out[:7] == [comb(heads, 3), 0, 0, 0, 0, 0, 0]
    counts_normally(harp)
