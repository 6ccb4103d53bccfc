"""harp_build_csr against numpy on messy edge lists: repeats in both directions, self-loops, rows at the edges of the
sort tiers before and after dropping repeats, hubs over one and several bitmap windows, lists that run along one
vertex, clean lists, bad ids."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
TIERS = (1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 64, 65, 128, 129, 256, 257, 512, 513, 1023, 1024, 1025, 2300, 4095, 4096, 4097,
         12000)


@pytest.fixture(scope="module")
def harp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_12074_gb300 import _build, harp as H
    _build.build()
    H.lib()
    return H


def device_array(ptr, count, typestr):
    class View:
        __cuda_array_interface__ = {"shape": (count,), "typestr": typestr, "data": (ptr, False), "version": 3}
    return torch.as_tensor(View(), device="cuda").cpu().numpy()


def expect(n, s, d):
    keep = s != d
    a, b = s[keep].astype(np.int64), d[keep].astype(np.int64)
    keys = np.unique(np.concatenate([a * n + b, b * n + a]))
    off = np.concatenate([[0], np.cumsum(np.bincount(keys // n, minlength=n))]).astype(np.int64)
    return off, (keys % n).astype(np.int32)


def stars(n, repeats, rng):
    """A star per tier size on shared random leaves, each edge listed `repeats` times in random directions."""
    s, d = [], []
    for k, size in enumerate(TIERS):
        leaves = rng.choice(np.arange(len(TIERS), n), size, replace=False)
        for r in range(repeats):
            hub = np.full(size, k)
            flip = rng.random(size) < 0.5
            s.append(np.where(flip, hub, leaves))
            d.append(np.where(flip, leaves, hub))
    s, d = np.concatenate(s), np.concatenate(d)
    return s, d


def cases():
    rng = np.random.RandomState(5)
    yield "stars", 20_000, *stars(20_000, 1, rng), True
    yield "stars_repeated", 20_000, *stars(20_000, 3, rng), True
    yield "two_windows", 1_700_000, *stars(1_700_000, 2, rng), True
    s, d = rng.randint(0, 900, 40_000), rng.randint(0, 900, 40_000)  # many repeats, self-loops
    yield "messy", 900, s, d, True
    yield "along_one_vertex", 30_000, np.zeros(29_999, np.int64), np.arange(1, 30_000), False
    yield "path", 1_000, np.arange(999), np.arange(1, 1000), False
    yield "loops_only", 5, np.array([1, 2, 3]), np.array([1, 2, 3]), False
    yield "one_edge_often", 3, np.full(5_000, 2), np.full(5_000, 0), False


CASES = {c[0]: c[1:] for c in cases()}


@pytest.mark.parametrize("device", [False, True], ids=["host", "device"])
@pytest.mark.parametrize("name", CASES)
def test_build(harp, name, device):
    n, s, d, shuffle = CASES[name]
    s, d = s.astype(np.int32), d.astype(np.int32)
    if shuffle:
        order = np.random.RandomState(6).permutation(s.size)
        s, d = s[order], d[order]
    off, cols = expect(n, s, d)
    args = (torch.from_numpy(s).cuda(), torch.from_numpy(d).cuda()) if device else (s, d)
    g = harp.harp_build_csr(n, *args)
    info = g.info()
    p_off, p_cols = harp.harp_csr_arrays(g)
    assert info["n"] == n and info["m"] == cols.size // 2 and info["max_degree"] == np.diff(off).max()
    assert np.array_equal(device_array(p_off, n + 1, "<i8"), off)
    if cols.size:
        assert np.array_equal(device_array(p_cols, cols.size, "<i4"), cols)
    g.close()


@pytest.mark.parametrize("n,pair", [(4, (0, 4)), (4, (-1, 2)), (4, (7, 7)), (0, (0, 0))])
def test_bad_ids(harp, n, pair):
    s, d = np.array([0, pair[0]], np.int32), np.array([1, pair[1]], np.int32)
    with pytest.raises(harp.HarpError) as e:
        harp.harp_build_csr(n, s, d)
    assert e.value.status == harp.HARP_EINVAL
