"""The hash tiers of the wedge pass against the CPU oracle, bit-exact: roots counted without a table (W <= 32), with
more lower neighbours than lanes, one-word and two-word tables, chunks of consecutive roots over many graphs."""
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


def leafy_cycle(length, leaves):
    """A cycle whose vertices carry `leaves` leaves each: many lower neighbours, few wedges of degree >= 2."""
    i = np.arange(length, dtype=np.int32)
    own = np.repeat(i, leaves)
    leaf = (length + np.arange(own.size)).astype(np.int32)
    return length + own.size, np.concatenate([i, own]), np.concatenate([(i + 1) % length, leaf]).astype(np.int32)


def among_isolated(g, n):
    """g's vertices spread over n ids (the table layout depends on the number of vertices)."""
    ids = np.linspace(0, n - 1, g.n).astype(np.int32)
    return n, ids[g.src], ids[g.dst]


CASES = {
    "leafy4x40": lambda: leafy_cycle(4, 40),
    "leafy4x33": lambda: leafy_cycle(4, 33),
    "leafy5x100": lambda: leafy_cycle(5, 100),
    "rgg30001": lambda: (lambda g: (g.n, g.src, g.dst))(graphgen.rgg(30001, 17.0, 3)),
    "er20000": lambda: (lambda g: (g.n, g.src, g.dst))(graphgen.er(20000, 40.0, 4)),
    "ba_in_2.2M": lambda: among_isolated(graphgen.ba(6000, 8, 5), 2_200_000),
    "ba_in_8.5M": lambda: among_isolated(graphgen.ba(6000, 8, 6), 8_500_000),
}


@pytest.mark.parametrize("name", CASES)
def test_tier_counts(harp, name):
    n, s, d = CASES[name]()
    g = harp.harp_build_csr(n, s, d)
    try:
        got = harp.harp_count4(g).tolist()
    finally:
        g.close()
    ids, inv = np.unique(np.concatenate([s, d]), return_inverse=True)  # the oracle without the isolated vertices
    assert got == O.count4_combo(ids.size, inv[:s.size].astype(np.int32), inv[s.size:].astype(np.int32)).tolist()


@pytest.mark.parametrize("copies", [3, 700])
def test_many_small_members(harp, copies):
    base = [leafy_cycle(4, 40), leafy_cycle(3, 2), (2, np.array([0], np.int32), np.array([1], np.int32))]
    base += [(g.n, g.src, g.dst) for g in (graphgen.rgg(300, 12.0, 8), graphgen.er(90, 9.0, 9), graphgen.ba(200, 5, 10))]
    want = [O.count4_combo(*m).tolist() for m in base]
    hs = [harp.harp_build_csr(*m) for m in base]
    b = harp.harp_batch_create(hs * copies)
    try:
        assert harp.harp_batch_count(b).tolist() == want * copies
    finally:
        b.close()
        for h in hs:
            h.close()
