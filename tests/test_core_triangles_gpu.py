"""Triangle rows read from the core's bitmaps against the CPU oracle, bit-exact: anchors whose lists lie all in the
core and partly below it, at the sizes where the modes and the tiles of a row change, with and without reuse of the
rows (without, every row is walked)."""
import numpy as np
import pytest

import graphgen
import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES = (33, 40, 41, 63, 64, 65, 97, 255, 256, 257, 271, 272, 273, 511, 512, 513)
CORE, LOW = 2040, 4000


def ladder(below):
    """A random core; per size an anchor adjacent to `size` vertices, `below` of them outside the core."""
    core = graphgen.er(CORE, 640.0, 11)
    rng = np.random.default_rng(7)
    low = graphgen.er(LOW, 20.0, 12)
    src, dst = [core.src, low.src + CORE], [core.dst, low.dst + CORE]
    # joins between the two parts, so that rows of either side have members of the list
    src.append(rng.integers(0, CORE, 30000).astype(np.int32))
    dst.append(rng.integers(CORE, CORE + LOW, 30000).astype(np.int32))
    n = CORE + LOW
    for size in SIZES:
        k = min(below, size)
        dst.append(np.concatenate([rng.choice(CORE, size - k, replace=False), CORE + rng.choice(LOW, k, replace=False)]))
        src.append(np.full(size, n))
        n += 1
    return n, np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)


@pytest.mark.parametrize("below", (0, 1, 16, 33))
def test_rows_from_the_core(below):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_12074_gb300 import harp as H

    n, s, d = ladder(below)
    want = O.count4_combo(n, s, d).tolist()
    g = H.harp_build_csr(n, s, d)
    try:
        assert H.harp_count4(g).tolist() == want
        p = H.harp_plan()
        p.version = H.HARP_ABI_VERSION
        p.flags = H.HARP_PLAN_NO_REUSE
        assert H.harp_count4(g, p).tolist() == want
    finally:
        g.close()
