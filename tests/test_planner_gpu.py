"""The basis that harp_select_anchors names, on graphs where one of the two was measured at least 7 % faster (microseconds
of a waiting count with the triangle-wedge and the literal basis in the comments; medians of 21)."""
import pytest

import graphgen

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = {
    "ba_300_3": (lambda: graphgen.ba(300, 3, 21), True),        # 96, 76
    "er_300_6": (lambda: graphgen.er(300, 6, 1), True),         # 81, 75
    "er_1000_3": (lambda: graphgen.er(1000, 3, 3), True),       # 83, 73
    "er_1000_10": (lambda: graphgen.er(1000, 10, 3), True),     # 101, 87
    "er_3000_2": (lambda: graphgen.er(3000, 2, 2), True),       # 100, 91
    "rmat_9_2": (lambda: graphgen.rmat(9, 2, seed=1), False),   # 100, 109
    "er_3000_16": (lambda: graphgen.er(3000, 16, 2), False),    # 124, 135
    "ba_3000_10": (lambda: graphgen.ba(3000, 10, 3), False),    # 155, 197
    "rgg_3000_10": (lambda: graphgen.rgg(3000, 10, 12), False),  # 112, 153
    "er_10000_4": (lambda: graphgen.er(10000, 4, 2), False),    # 111, 150
    "ba_22000_4": (lambda: graphgen.ba(22000, 4, 3), False),    # 189, 376
    "er_80000_4": (lambda: graphgen.er(80000, 4, 2), False),    # 203, 548
    "rmat_13_8": (lambda: graphgen.rmat(13, 8, seed=1), False),  # 206, 681
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
def test_basis(harp, name):
    make, literal = CASES[name]
    g = make()
    csr = harp.harp_build_csr(g.n, g.src, g.dst)
    p = harp.harp_select_anchors(csr)
    csr.close()
    assert (p.basis == harp.HARP_BASIS_LITERAL) == literal == (p.est_cost_lit < p.est_cost_tw)
