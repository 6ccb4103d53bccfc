"""harp_build_csr where hub rows wait for the host's choice between bitmaps and a radix sort (more than 2^18 entry reads, or
ids of more than four windows), against numpy: rows on both sides of both lines, either sort, repeats, and rows of
every other tier beside."""
import os
import sys

import numpy as np
import pytest

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
from test_build_gpu import device_array, expect, stars  # noqa: E402

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

WINDOW = 32 * 50_176  # ids of one bitmap window


def long_rows(n, sizes, repeats, rng):
    """A row per size (entries, repeats included) and the small tiers' stars."""
    s, d = stars(n, 1, rng) if n > 100_000 else (np.zeros(0, np.int64), np.zeros(0, np.int64))
    parts = [(s, d)]
    for k, size in enumerate(sizes):
        hub = n - 1 - k
        leaves = rng.randint(0, n - len(sizes), (size + repeats - 1) // repeats)
        other = np.tile(leaves, repeats)[:size]
        parts.append((np.full(size, hub), other))
    s, d = (np.concatenate(x) for x in zip(*parts))
    flip = rng.random(s.size) < 0.5
    return np.where(flip, s, d), np.where(flip, d, s)


CASES = {
    "line_one_window": (300_000, (1 << 18, (1 << 18) + 1, 4097, 400_000), 1),
    "line_two_windows": (WINDOW + 1, (1 << 17, (1 << 17) + 1, 5000), 1),
    "repeats": (20_000, (300_000, 262_145, 280_000), 20),
    "four_windows": (4 * WINDOW, (4097, 1 << 16, (1 << 16) + 1), 1),
    "five_windows": (4 * WINDOW + 1, (4096, 4097, 9000, 70_000), 2),
    "five_windows_radix": (4 * WINDOW + 1, (4097, 1_500_000), 2),
    "bitmap_for_all": (40_000, (300_000,) * 30, 20),
}


@pytest.fixture(scope="module")
def harp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_12074_gb300 import _build, harp as H
    _build.build()
    H.lib()
    return H


@pytest.mark.parametrize("name", CASES)
def test_build(harp, name):
    n, sizes, repeats = CASES[name]
    s, d = long_rows(n, sizes, repeats, np.random.RandomState(7))
    off, cols = expect(n, s, d)
    g = harp.harp_build_csr(n, torch.from_numpy(s.astype(np.int32)).cuda(), torch.from_numpy(d.astype(np.int32)).cuda())
    info = g.info()
    p_off, p_cols = harp.harp_csr_arrays(g)
    assert info["m"] == cols.size // 2 and info["max_degree"] == np.diff(off).max()
    assert np.array_equal(device_array(p_off, n + 1, "<i8"), off)
    assert np.array_equal(device_array(p_cols, cols.size, "<i4"), cols)
    g.close()


@pytest.mark.parametrize("leaves", [261_000, 263_000])
def test_star_without_repeats(harp, leaves):
    """Nothing is dropped: the sorted rows are the columns."""
    n = leaves + 1
    s, d = np.zeros(leaves, np.int32), np.random.RandomState(8).permutation(np.arange(1, n)).astype(np.int32)
    g = harp.harp_build_csr(n, s, d)
    p_off, p_cols = harp.harp_csr_arrays(g)
    off, cols = expect(n, s, d)
    assert np.array_equal(device_array(p_off, n + 1, "<i8"), off)
    assert np.array_equal(device_array(p_cols, cols.size, "<i4"), cols)
    assert harp.harp_count4(g).tolist()[0] == leaves * (leaves - 1) * (leaves - 2) // 6
    g.close()


def test_bad_id_beside_long_rows(harp):
    s = np.zeros(300_001, np.int32)
    d = np.arange(1, 300_002, dtype=np.int32)
    with pytest.raises(harp.HarpError) as e:
        harp.harp_build_csr(300_001, s, d)
    assert e.value.status == harp.HARP_EINVAL
