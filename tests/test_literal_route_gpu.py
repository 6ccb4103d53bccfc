"""Which edge pass a literal count takes: staged frontiers where a vertex has enough edges to pay for a block's turn, the
pass by edges on sparse graphs, on both sides of each line of the rule; and what harp_reuse_stats counts in either.
Copies of K_{2,3} beside a star: in the staged pass an edge's request and 4 of a copy's 6 requests for the two hubs'
frontier are answered by its counters, whatever the signature cache holds; the pass by edges has nothing but the
cache."""
from math import comb

import numpy as np
import pytest

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


def bicliques_and_star(n, leaves):
    """K_{2,3} on every five vertices, then a star of so many leaves on the last ones."""
    copies = (n - leaves - 1) // 5 if leaves else n // 5
    base = 5 * np.arange(copies, dtype=np.int64)[:, None]
    src = (base + np.array([0, 0, 0, 1, 1, 1])).ravel()
    dst = (base + np.array([2, 3, 4, 2, 3, 4])).ravel()
    src = np.concatenate([src, np.full(leaves, n - 1)])
    dst = np.concatenate([dst, n - 1 - np.arange(1, leaves + 1)])
    return copies, src.astype(np.int32), dst.astype(np.int32)


# mean degree about 2.4: staged up to 2,048 vertices; then mean^2 + 0.3 d_max >= min(15 + n / 1000, 41) while two blocks
# fit an SM (n <= 45,511), mean^2 + 0.15 d_max >= 95 up to 90,000 vertices
CASES = [(2048, 0, True), (2049, 0, False), (10_000, 55, False), (10_000, 75, True), (40_000, 110, False),
         (40_000, 125, True), (45_500, 125, True), (45_600, 125, False), (80_000, 0, False), (80_000, 560, False),
         (80_000, 620, True), (90_000, 620, True), (90_001, 620, False)]


@pytest.mark.parametrize("n,leaves,staged", CASES)
def test_route(harp, n, leaves, staged):
    copies, src, dst = bicliques_and_star(n, leaves)
    want = [2 * copies + comb(leaves, 3), 0, 0, 3 * copies, 0, 0]
    seen = {}
    g = harp.harp_build_csr(n, src, dst)
    for slots, min_deg in ((0, 0), (6, 0), (0, 3)):
        plan = harp.harp_plan()
        plan.version, plan.basis, plan.lit_cache_log2 = harp.HARP_ABI_VERSION, harp.HARP_BASIS_LITERAL, slots
        plan.lit_cache_min_deg = min_deg
        assert harp.harp_count4(g, plan).tolist() == want
        seen[slots, min_deg] = harp.harp_reuse_stats(g)
    g.close()
    # requests: one per edge in the first pass, one per edge and 6 per copy in the second, two per edge in the third
    edges = 6 * copies + leaves
    assert {lookups for lookups, _ in seen.values()} == {4 * edges + 6 * copies}
    full, tiny, hubs = (seen[k][1] for k in ((0, 0), (6, 0), (0, 3)))
    if staged:
        assert full == 3 * edges + 4 * copies
        assert edges + 4 * copies <= tiny <= edges + 4 * copies + 128  # the third pass finds at most 64 edges kept
        assert hubs == 4 * copies
    else:  # of the 6, those made before the first is kept miss
        assert 3 * edges <= full <= 3 * edges + 5 * copies
        assert tiny <= 1000  # what 64 slots can answer
        assert hubs <= 5 * copies
