"""The streams that host code uses, without a GPU: the library's objects linked with a fake CUDA runtime
(fake_cudart.c) in which kernels do nothing and every enqueued operation is recorded."""
import ctypes
import glob
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
GREATEST = -5  # the fake's priorities: 0 .. -5


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_2607_12074_gb300 import _build
    nvcc = shutil.which(_build.nvcc())
    if not nvcc or not shutil.which("gcc"):
        pytest.skip("needs nvcc and gcc to link the library with the fake runtime")
    _build.build()
    out = tmp_path_factory.mktemp("fake")
    obj, lib = str(out / "fake_cudart.o"), str(out / "libharp_fake.so")
    include = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    subprocess.run(["gcc", "-O1", "-fPIC", "-I", include, "-c", os.path.join(HERE, "fake_cudart.c"), "-o", obj], check=True)
    # -Bsymbolic: another CUDA runtime that the process has loaded (torch's) must not take the fake's place
    subprocess.run([nvcc, *_build.ARCH, "-shared", "-cudart", "none", "-Xlinker", "-Bsymbolic", "-o", lib,
                    *glob.glob(os.path.join(_build.BUILD, "*.cu.o")), obj], check=True)
    L = ctypes.CDLL(lib)
    L.fake_launches.restype = L.fake_calls.restype = ctypes.c_long
    L.harp_status_str.restype = ctypes.c_char_p
    return L


def submit(L, server, edges):
    n = edges + 1
    src, dst = np.arange(edges, dtype=np.int32), np.arange(1, n, dtype=np.int32)
    ticket = ctypes.c_uint64()
    ptr = ctypes.POINTER(ctypes.c_int32)
    assert L.harp_submit(server, ctypes.c_int64(n), ctypes.c_int64(edges), src.ctypes.data_as(ptr), dst.ctypes.data_as(ptr),
                         ctypes.byref(ticket)) == 0
    counts = (ctypes.c_uint64 * 6)()
    assert L.harp_wait(server, ticket, counts, ctypes.c_double(20_000)) == 0


def test_server_lanes_keep_to_their_priority(fake):
    """CSR build, union and count of a small request run at the small lane's priority, those of a large one at the
    lowest."""
    L = fake
    server = ctypes.c_void_p()
    assert L.harp_server_create(None, ctypes.byref(server)) == 0
    try:
        before = {p: L.fake_launches(p) for p in (0, GREATEST)}
        submit(L, server, 1000)
        small = {p: L.fake_launches(p) for p in (0, GREATEST)}
        assert small[0] == before[0] and small[GREATEST] > before[GREATEST]
        submit(L, server, 65_537)
        large = {p: L.fake_launches(p) for p in (0, GREATEST)}
        assert large[0] > small[0] and large[GREATEST] == small[GREATEST]
    finally:
        L.harp_server_destroy(server)


def build(L, n, m, stream):
    """A handle of n vertices and m edges, all in the fake's word: no repeats, largest degree 40."""
    L.fake_answer((ctypes.c_uint64 * 8)(0, 40, 2 * m, 0, 0, 0, 0, 0), ctypes.c_size_t(64))
    src = np.zeros(m, np.int32)
    ptr = src.ctypes.data_as(ctypes.POINTER(ctypes.c_int32))
    g = ctypes.c_void_p()
    assert L.harp_build_csr(ctypes.c_int64(n), ctypes.c_int64(m), ptr, ptr, 0, stream, ctypes.byref(g)) == 0
    return g


@pytest.mark.parametrize("literal", [False, True], ids=["triangle_wedge", "literal"])
def test_side_streams_are_joined_where_a_call_fails(fake, literal):
    """Whichever runtime call of a count fails, the handle's stream waits for all work given to the side streams, so
    that freeing the handle (ordered on its stream) cannot overtake it."""
    from paper_2607_12074_gb300 import harp as H
    L = fake
    p = H.harp_plan()
    p.version, p.basis = H.HARP_ABI_VERSION, H.HARP_BASIS_LITERAL if literal else H.HARP_BASIS_TRIANGLE_WEDGE
    plan = ctypes.byref(p)
    g = build(L, 2000, 9000, None)
    counts = (ctypes.c_uint64 * 6)()
    assert L.harp_count4(g, plan, counts) == 0
    open_before = L.fake_unjoined(None)
    L.fake_fail_at(ctypes.c_long(-1))
    assert L.harp_count4(g, plan, counts) == 0
    calls = L.fake_calls()
    assert calls >= 20
    for k in range(calls):
        L.fake_fail_at(ctypes.c_long(k))
        status = L.harp_count4(g, plan, counts)
        assert status != 0, k
        assert L.fake_unjoined(None) == open_before, k
    L.fake_fail_at(ctypes.c_long(-1))
    assert L.harp_count4(g, plan, counts) == 0
    L.harp_csr_free(g)


@pytest.mark.parametrize("literal", [False, True], ids=["triangle_wedge", "literal"])
@pytest.mark.parametrize("priority", [0, -2, GREATEST])
def test_side_streams_have_the_priority_of_the_handles_stream(fake, priority, literal):
    from paper_2607_12074_gb300 import harp as H
    L = fake
    p = H.harp_plan()
    p.version, p.basis = H.HARP_ABI_VERSION, H.HARP_BASIS_LITERAL if literal else H.HARP_BASIS_TRIANGLE_WEDGE
    stream = ctypes.c_void_p()
    assert L.cudaStreamCreateWithPriority(ctypes.byref(stream), 1, priority) == 0
    before = [L.fake_launches(q) for q in range(0, GREATEST - 1, -1)]
    g = build(L, 2000, 9000, stream)
    counts = (ctypes.c_uint64 * 6)()
    assert L.harp_count4(g, ctypes.byref(p), counts) == 0
    L.harp_csr_free(g)
    after = [L.fake_launches(q) for q in range(0, GREATEST - 1, -1)]
    assert [q for q in range(6) if after[q] > before[q]] == [-priority]
