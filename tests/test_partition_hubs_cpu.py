"""The host rank graph where the hubs have consecutive ids (a bucket of ids taken by every host thread), and the
triangle blocks' scratch, which follows the largest out-degree of the graph at hand."""
import numpy as np
import pytest

import graphgen
from test_partition_plan_cpu import check_tiling, rank_graph_reference

H = pytest.importorskip("paper_2607_12074_gb300.harp")


@pytest.mark.parametrize("first", (0, 30_000))
@pytest.mark.parametrize("hubs", (1, 40))
def test_hubs_of_close_ids(hubs, first):
    n, m = 50_000, 900_000
    rng = np.random.default_rng(hubs)
    src = rng.integers(first, first + hubs, m).astype(np.int32)  # every edge at a hub, many of them repeated
    dst = rng.integers(0, n, m).astype(np.int32)
    src[m // 2:], dst[m // 2:] = dst[m // 2:].copy(), src[m // 2:].copy()
    rank, off, cols = H.harp_rank_csr_host(n, src, dst)
    want = rank_graph_reference(n, src, dst)
    for got, ref in zip((rank, off, cols), want):
        assert np.array_equal(got, ref)


def test_scratch_follows_the_out_degrees():
    # 1.5 million edges allow an out-degree above 1,024 (318 MB of scratch); this graph's stays below 64
    g = graphgen.er(100_000, 30.0, 3)
    st, tri, wedge = H.harp_partition_plan(g.n, g.src, g.dst, 128 << 20)
    check_tiling(g.n, tri, wedge)
    assert st["tri_blocks"] == 1 and st["device_peak_bytes"] <= 128 << 20
