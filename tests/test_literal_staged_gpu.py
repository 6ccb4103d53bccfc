"""The literal basis's edge pass with staged frontiers against the CPU oracle, bit-exact: the largest staged graph and
the smallest that is not, hubs among leaves, sparse graphs whose counters are cleared by a second walk, dense ones
cleared as a whole, every cache size and admission, and without reuse (the unstaged pass)."""
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


def padded(g, n):
    """g with isolated vertices up to n."""
    return n, g.src, g.dst


def wheel_with_leaves(rim, leaves):
    i = np.arange(rim, dtype=np.int32)
    hub = np.full(rim + leaves, rim, np.int32)
    out = np.concatenate([i, rim + 1 + np.arange(leaves, dtype=np.int32)])
    return rim + 1 + leaves, np.concatenate([i, hub]).astype(np.int32), np.concatenate([(i + 1) % rim, out]).astype(np.int32)


CASES = {
    "staged_n90000": lambda: padded(graphgen.ba(3000, 5, 1), 90000),
    "unstaged_n90001": lambda: padded(graphgen.ba(3000, 5, 1), 90001),
    "sparse_rgg": lambda: padded(graphgen.rgg(30000, 8.0, 2), 30000),
    "dense_er": lambda: padded(graphgen.er(700, 120.0, 3), 701),
    "wheel": lambda: wheel_with_leaves(1000, 5001),
    "rmat12": lambda: padded(graphgen.rmat(12, 16, seed=4), 4096),
}


@pytest.mark.parametrize("kw", [{}, {"lit_cache_log2": 6}, {"lit_cache_min_deg": 12}, {"flags": 2}],
                         ids=["default", "64_slots", "min_degree_12", "no_reuse"])
@pytest.mark.parametrize("name", CASES)
def test_literal(harp, name, kw):
    n, s, d = CASES[name]()
    plan = harp.harp_plan()
    plan.version, plan.basis = harp.HARP_ABI_VERSION, harp.HARP_BASIS_LITERAL
    for k, v in kw.items():
        setattr(plan, k, v)
    g = harp.harp_build_csr(n, s, d)
    try:
        got = harp.harp_count4(g, plan).tolist()
        lookups, hits = harp.harp_reuse_stats(g)
    finally:
        g.close()
    assert got == O.count4_combo(n, s, d).tolist()
    assert hits < lookups and (hits == 0 or not kw.get("flags"))
