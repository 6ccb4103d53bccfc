"""The basis that harp_select_anchors names, on graphs where one of the two was measured at least 7 % faster (microseconds
of a waiting count with the triangle-wedge and the literal basis in the comments; medians of 21)."""
import pytest

import graphgen

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = {
    "ba_300_3": (lambda: graphgen.ba(300, 3, 21), True),        # 98, 84
    "er_300_6": (lambda: graphgen.er(300, 6, 1), True),         # 84, 76
    "er_1000_3": (lambda: graphgen.er(1000, 3, 3), True),       # 84, 77
    "er_3000_2": (lambda: graphgen.er(3000, 2, 2), True),       # 101, 89
    "rmat_9_2": (lambda: graphgen.rmat(9, 2, seed=1), False),   # 96, 120
    "rgg_1000_8": (lambda: graphgen.rgg(1000, 8, 3), False),    # 90, 98
    "er_3000_8": (lambda: graphgen.er(3000, 8, 2), False),      # 113, 127
    "ba_3000_4": (lambda: graphgen.ba(3000, 4, 3), False),      # 132, 143
    "rgg_3000_10": (lambda: graphgen.rgg(3000, 10, 12), False),  # 116, 166
    "er_10000_4": (lambda: graphgen.er(10000, 4, 2), False),    # 114, 151
    "ba_22000_4": (lambda: graphgen.ba(22000, 4, 3), False),    # 190, 401
    "er_80000_4": (lambda: graphgen.er(80000, 4, 2), False),    # 202, 547
    "rmat_13_8": (lambda: graphgen.rmat(13, 8, seed=1), False),  # 202, 805
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
