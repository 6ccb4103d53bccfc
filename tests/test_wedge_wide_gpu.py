"""The wide hash tier of the wedge pass (2,048 < W <= 16,384, several windows) against the CPU oracle, bit-exact: work
around its limits, as many lower neighbours as its counts hold and one more, tables cut to the root, and the same
roots through the windows."""
import numpy as np
import pytest

import graphgen
import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def with_path(n, s, d, total):
    """Beside a path (another band of degrees), among isolated vertices."""
    i = np.arange(n, n + 999)
    return total, np.concatenate([s, i]).astype(np.int32), np.concatenate([d, i + 1]).astype(np.int32)


def bipartite(a, b):
    s, d = np.meshgrid(np.arange(a), a + np.arange(b), indexing="ij")
    return a + b, s.ravel(), d.ravel()


def of(g):
    return g.n, g.src, g.dst


CASES = {
    "er6000x110": lambda: with_path(*of(graphgen.er(6000, 110.0, 3)), 30_000),
    "er4000x180": lambda: with_path(*of(graphgen.er(4000, 180.0, 4)), 30_000),
    "er2600x230_in_4.2M": lambda: with_path(*of(graphgen.er(2600, 200.0, 5)), 4_194_400),
    "er2600x230_in_4.1M": lambda: with_path(*of(graphgen.er(2600, 200.0, 5)), 4_194_200),
    "K5x1023": lambda: with_path(*bipartite(5, 1023), 30_000),
    "K5x1024": lambda: with_path(*bipartite(5, 1024), 30_000),
    "K5x1025": lambda: with_path(*bipartite(5, 1025), 30_000),
    "K9x1024": lambda: with_path(*bipartite(9, 1024), 30_000),   # W = 8,192
    "K10x1024": lambda: with_path(*bipartite(10, 1024), 30_000),
    "K17x1024": lambda: with_path(*bipartite(17, 1024), 30_000),  # W = 16,384
    "K18x1024": lambda: with_path(*bipartite(18, 1024), 30_000),
}


@pytest.mark.parametrize("name", CASES)
def test_wide_roots(name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_12074_gb300 import harp as H

    n, s, d = CASES[name]()
    ids, inv = np.unique(np.concatenate([s, d]), return_inverse=True)  # the oracle without the isolated vertices
    want = O.count4_combo(ids.size, inv[:s.size].astype(np.int32), inv[s.size:].astype(np.int32)).tolist()
    g = H.harp_build_csr(n, s, d)
    try:
        for flags, most in ((0, 0), (H.HARP_PLAN_NO_BAND_MERGE, 0), (H.HARP_PLAN_NO_BAND_MERGE, 2047)):
            p = H.harp_plan()
            p.version = H.HARP_ABI_VERSION
            p.flags, p.c4_cta_max_work = flags, most
            assert H.harp_count4(g, p).tolist() == want
    finally:
        g.close()
