"""The device build where counters are spread over the id's low bits (from 16,384 vertices) and rows are closed up by
runs of columns: hubs of neighbouring ids, repeats everywhere, long stretches of isolated vertices."""
import numpy as np
import pytest

from test_build_gpu import device_array, expect, harp  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", (33, 16383, 16384, 16385, 16415, 40001))
@pytest.mark.parametrize("m", (40, 5000, 300_000))
def test_hubs_of_close_ids_and_empty_rows(harp, n, m):  # noqa: F811
    rng = np.random.default_rng(n + m)
    hub = (n * rng.random(m) ** 6).astype(np.int64)          # most pairs at the lowest ids
    other = n - 1 - (n * rng.random(m) ** 3 / 4).astype(np.int64)  # the middle stays isolated
    s, d = np.concatenate([hub, other[: m // 3]]), np.concatenate([other, hub[: m // 3]])
    off, cols = expect(n, s, d)
    g = harp.harp_build_csr(n, s.astype(np.int32), d.astype(np.int32))
    try:
        info = g.info()
        assert (info["n"], info["m"]) == (n, len(cols) // 2)
        p_off, p_cols = harp.harp_csr_arrays(g)
        assert np.array_equal(device_array(p_off, n + 1, "<i8"), off)
        assert np.array_equal(device_array(p_cols, len(cols), "<i4"), cols)
    finally:
        g.close()
