"""The tiers of the orbit outputs at sizes the other tests do not reach, against closed forms: heavy roots with
16-bit and 32-bit windows and with global counters, middle roots, hub rows, anchors of out-degree above 1024."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
C = math.comb


@pytest.fixture(scope="module")
def harp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_12074_gb300 import _build, harp as H
    _build.build()
    H.lib()
    return H


@pytest.mark.parametrize("leaves,isolated", [(600, 0), (3001, 0), (70001, 0), (3001, 400_000)],
                         ids=["middle", "window16", "window32", "global"])
def test_two_hubs(harp, leaves, isolated):
    """K_{2,leaves}: wedge work `leaves` at the top hub; every 4-subset is a star, a 4-cycle or not connected."""
    N, n = leaves, leaves + 2 + isolated
    leaf = np.arange(2, N + 2, dtype=np.int32)
    g = harp.harp_build_csr(n, np.concatenate([0 * leaf, 0 * leaf + 1]), np.concatenate([leaf, leaf]))
    v, e = harp.harp_count4_orbits(g), harp.harp_count4_edge_orbits(g)
    g.close()
    want = np.zeros((n, harp.HARP_NORBITS), np.uint64)
    want[:2, harp.ORBITS.index("star_center")] = C(N, 3)
    want[:2, harp.ORBITS.index("cycle")] = C(N, 2)
    want[2:N + 2, harp.ORBITS.index("star_leaf")] = 2 * C(N - 1, 2)
    want[2:N + 2, harp.ORBITS.index("cycle")] = N - 1
    assert np.array_equal(v, want)
    want = np.zeros((2 * N, harp.HARP_NEDGE_ORBITS), np.uint64)
    want[:, harp.EDGE_ORBITS.index("star_edge")] = C(N - 1, 2)
    want[:, harp.EDGE_ORBITS.index("cycle_edge")] = N - 1
    assert np.array_equal(e, want)


@pytest.mark.parametrize("k", [33, 300, 600, 1030], ids=lambda k: f"K{k}")
def test_cliques(harp, k):
    """K_k: out-degrees up to k - 1 (every triangle tier, 1029 included), only 4-cliques."""
    i, j = np.triu_indices(k, 1)
    g = harp.harp_build_csr(k, i.astype(np.int32), j.astype(np.int32))
    v, e = harp.harp_count4_orbits(g), harp.harp_count4_edge_orbits(g)
    g.close()
    assert (v[:, :-1] == 0).all() and (v[:, -1] == C(k - 1, 3)).all()
    assert (e[:, :-1] == 0).all() and (e[:, -1] == C(k - 2, 2)).all()
