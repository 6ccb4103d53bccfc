"""Counts on streams that the caller made: handles on streams of each priority, and harp_count4_async and
harp_count4_noalloc captured into the caller's own CUDA graph and replayed."""
import numpy as np
import pytest

import graphgen
import oracle as O

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


@pytest.mark.parametrize("priority", [0, -1, -5])
def test_handle_on_a_priority_stream(harp, priority):
    stream = torch.cuda.Stream(priority=priority)
    for g in (graphgen.ba(2000, 4, 1), graphgen.rmat(13, 16, seed=2)):
        csr = harp.harp_build_csr(g.n, g.src, g.dst, stream)
        want = O.count4_combo(g.n, g.src, g.dst).tolist()
        plan = harp.harp_plan()
        plan.version, plan.basis = harp.HARP_ABI_VERSION, harp.HARP_BASIS_LITERAL
        for _ in range(3):
            assert harp.harp_count4(csr).tolist() == want
            assert harp.harp_count4(csr, plan).tolist() == want
        csr.close()


GRAPHS = {"small": lambda: graphgen.ba(2000, 4, 1), "core": lambda: graphgen.rmat(15, 12, seed=3)}


@pytest.mark.parametrize("name", GRAPHS)
@pytest.mark.parametrize("noalloc", [False, True], ids=["async", "noalloc"])
def test_captured_by_the_caller(harp, name, noalloc):
    g = GRAPHS[name]()
    want = O.count4_combo(g.n, g.src, g.dst).tolist()
    csr = harp.harp_build_csr(g.n, g.src, g.dst)
    info, (off, cols) = csr.info(), harp.harp_csr_arrays(csr)
    out = torch.zeros(16, dtype=torch.int64, device="cuda")

    def enqueue(stream):
        if noalloc:
            harp.harp_count4_noalloc(info["n"], info["m"], off, cols, out.data_ptr(), stream)
        else:
            harp.harp_count4_async(csr, out.data_ptr(), None, stream)

    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    enqueue(stream)  # the workspace, or the scratch's address, is made outside the capture
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        enqueue(stream)
    for _ in range(3):
        out.fill_(-1)
        graph.replay()
        torch.cuda.synchronize()
        got = out.cpu().numpy().view(np.uint64)
        assert got[:6].tolist() == want and got[6] == 0
    csr.close()
