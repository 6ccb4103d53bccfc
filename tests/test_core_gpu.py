"""The wedge core (counters of the K highest ranks as bit planes) against the CPU oracle, bit-exact: every
counter width (x of degree below 16, 256, 65536 and above), x inside and below the core, core sizes from
1,024 up, rows split over a block's warps, and graphs with a core beside graphs without one in a batch."""
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


def clique_with_leaves(k, leaves):
    """K_k and one leaf on each of its first vertices: x, w and u all in the core, rows split over warps."""
    i, j = np.triu_indices(k, 1)
    src = np.concatenate([i, np.arange(leaves) % k])
    dst = np.concatenate([j, k + np.arange(leaves)])
    return k + leaves, src.astype(np.int32), dst.astype(np.int32)


def hubs_over_core(leaves, core):
    """Two hubs over `leaves` shared leaves and a random core: counts above 65,535 for the hub pair."""
    g = graphgen.er(core, 60.0, 5)
    n = 2 + core + leaves
    every = np.arange(2, n, dtype=np.int32)
    src = np.concatenate([g.src + 2, np.zeros(n - 2, np.int32), np.ones(n - 2, np.int32)])
    dst = np.concatenate([g.dst + 2, every, every])
    return n, src.astype(np.int32), dst.astype(np.int32)


def as_tuple(g):
    return g.n, g.src, g.dst


CASES = {
    "K1500+leaves": lambda: clique_with_leaves(1500, 3001),
    "hubs70000": lambda: hubs_over_core(70001, 4400),
    "rmat14x32": lambda: as_tuple(graphgen.rmat(14, 32, seed=3)),
    "rmat16": lambda: as_tuple(graphgen.rmat(16, 16, seed=4)),
    "rmat18": lambda: as_tuple(graphgen.rmat(18, 15, seed=5)),
    "chung_lu60001": lambda: as_tuple(graphgen.chung_lu(60001, 2.1, 3000.0, 40.0, 6)),
    "ba40001": lambda: as_tuple(graphgen.ba(40001, 8, 7)),
}


@pytest.fixture(scope="module")
def graphs():
    out = {}
    for name, make in CASES.items():
        n, s, d = make()
        out[name] = (n, s, d, O.count4_combo(n, s, d).tolist())
    return out


@pytest.mark.parametrize("name", CASES)
def test_core_counts(harp, graphs, name):
    n, s, d, want = graphs[name]
    g = harp.harp_build_csr(n, s, d)
    try:
        assert harp.harp_count4(g).tolist() == want
    finally:
        g.close()


def test_core_in_a_batch(harp, graphs):
    small = [as_tuple(graphgen.batch_graph(seed)) for seed in (1, 2, 3)]
    members = []
    for k, (n, s, d, want) in enumerate(graphs.values()):
        members.append((n, s, d, want))
        m = small[k % 3]
        members.append((*m, O.count4_combo(*m).tolist()))
    hs = [harp.harp_build_csr(n, s, d) for n, s, d, _ in members]
    b = harp.harp_batch_create(hs)
    try:
        for _ in range(2):
            assert harp.harp_batch_count(b).tolist() == [w for *_, w in members]
    finally:
        b.close()
        for h in hs:
            h.close()
