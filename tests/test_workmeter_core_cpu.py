"""The work meter's core pass against plain loops over a small graph, and the choice of the core."""
import os
import sys

import pytest

import graphgen
from paper_2607_12074_gb300 import workmeter

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
from test_workmeter_cpu import rank_adjacency  # noqa: E402


@pytest.mark.parametrize("K", [32, 128])
@pytest.mark.parametrize("make", [lambda: graphgen.rmat(9, 8, seed=2), lambda: graphgen.ba(400, 5, 3)], ids=["rmat", "ba"])
def test_core_bytes(make, K):
    g = make()
    adj = rank_adjacency(g.n, g.src, g.dst)
    G = workmeter.rank_space(g.n, g.src, g.dst)
    c0, KW = g.n - K, K // 32
    elements = words = rows = low = 0
    for x, row in enumerate(adj):
        if len(row) < 2:
            continue
        rows += len(row)
        for w in row:
            if w < c0:
                low += 1
                elements += sum(1 for u in adj[w] if u >= c0 and u > x)
            else:  # words of w's bitmap row that can hold a bit above x and w
                words += sum(1 for i in range(KW) if i >= (w - c0) // 32 and (x < c0 or i >= (x - c0 + 1) // 32))
    table = sum(4 * sum(1 for u in adj[w] if u > w) + 6 * (KW - ((w - c0) // 32 // 4 * 4)) for w in range(c0, g.n))
    got = workmeter.core_bytes(G, c0)
    assert got == {"bytes": table + 20 * g.n + 4 * rows + 8 * low + 4 * elements + 4 * words, "elements": elements,
                   "words": words}


def test_core_start():
    dense = graphgen.rmat(15, 16, seed=1)
    G = workmeter.rank_space(dense.n, dense.src, dense.dst)
    K = dense.n - workmeter.core_start(G)
    assert K in [1 << k for k in range(10, 15)]
    arcs = int(G["indptr"][-1] - G["indptr"][dense.n - K])
    assert G["deg"][dense.n - K] >= K // 64 and 4 * arcs >= G["m"] and 2 * K <= dense.n
    for g in (graphgen.rgg(60_000, 10.0, 1), graphgen.ba(2000, 4, 1)):  # no hubs; too few edges
        G = workmeter.rank_space(g.n, g.src, g.dst)
        assert workmeter.core_start(G) == g.n
        assert workmeter.meter(g.n, g.src, g.dst)["c4_core"]["bytes"] == 0
