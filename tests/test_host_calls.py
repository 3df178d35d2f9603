"""The library's host code on a stand-in for the CUDA runtime (tests/cuda_fake.cpp), without a GPU:
what it copies, allocates and launches, and in which order.

* the hub lists reach the device before the kernels that read them, on any stream;
* an allocation that fails is reported, leaks nothing, and leaves nothing that a kernel would read;
* a call that fails writes no out-parameter;
* a server's slots and copies take the memory that its budget is charged for;
* a graph without the mirror pass holds 8 bytes less per entry."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "cuda_fake.cpp")
N, DEGREE = 64, 40                                        # nodes of the test graph and their degree


@pytest.fixture(scope="module")
def lib():
    from paper_2508_01485_gb300 import build
    cxx = shutil.which("g++")
    try:
        if not cxx:
            raise RuntimeError("no host C++ compiler")
        build.build()
        objs = [os.path.join(build.OUT_DIR, os.path.basename(s).replace(".cu", ".o")) for s in build.sources()]
        if not all(os.path.exists(o) for o in objs):
            build.build(force=True)
    except RuntimeError as e:                             # no compiler on this machine
        pytest.skip(str(e))
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    out = os.path.join(HERE, "_build", "librs_fake.so")
    os.makedirs(os.path.dirname(out), exist_ok=True)
    tmp = out + ".%d.tmp" % os.getpid()
    subprocess.check_call([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", inc, "-o", tmp, SRC, *objs])
    os.replace(tmp, out)
    L = ctypes.CDLL(out)
    L.fake_stream.restype = ctypes.c_void_p
    L.fake_unordered.restype = ctypes.c_char_p
    L.fake_live_bytes.restype = ctypes.c_int64
    L.fake_fail_allocation.argtypes = [ctypes.c_int64]
    L.rs_last_error.restype = ctypes.c_char_p
    return L


def _ptr(a):
    return ctypes.c_void_p(a.ctypes.data)


class Calls:
    """The C calls on one stream of the stand-in, which is non-blocking like a server's or a
    torch side stream."""

    def __init__(self, lib):
        self.lib, self.s = lib, ctypes.c_void_p(lib.fake_stream())
        self.scores = np.zeros(N)

    def build(self, flags=0, n=N):
        nnz, off = n * DEGREE, np.arange(n + 1) * DEGREE
        cols, labels = np.zeros(nnz, np.int32), np.zeros(n, np.int32)
        g = ctypes.c_void_p()
        assert self.lib.rs_build_graph(ctypes.c_int64(n), ctypes.c_int64(nnz), _ptr(off), 1, _ptr(cols), _ptr(labels), 8, 0,
                                       flags, self.s, ctypes.byref(g)) == 0
        return g

    def score(self, g):
        return self.lib.rs_score(g, _ptr(self.scores), None, self.s)

    def remove(self, g, nodes=(0,), applied=None):
        v = np.asarray(nodes, np.int32)
        return self.lib.rs_apply_removals(g, _ptr(v), ctypes.c_int64(v.size), None, None, ctypes.c_int64(0),
                                          ctypes.byref(applied) if applied is not None else None, self.s)

    def server(self, graphs, slots=1, budget=1 << 40, mode=0):
        arr, srv = (ctypes.c_void_p * len(graphs))(*[g.value for g in graphs]), ctypes.c_void_p()
        assert self.lib.rs_server_create(arr, len(graphs), slots, ctypes.c_int64(budget), 4, mode, ctypes.byref(srv)) == 0
        return srv

    def tune(self, g, **fields):
        from paper_2508_01485_gb300 import _lib
        t = _lib.Tuning()
        assert self.lib.rs_get_tuning(g, ctypes.byref(t)) == 0
        for k, v in fields.items():
            setattr(t, k, v)
        return self.lib.rs_set_tuning(g, ctypes.byref(t), self.s)

    def used(self, srv):
        used = ctypes.c_int64()
        assert self.lib.rs_server_info(srv, None, ctypes.byref(used), None, None) == 0
        return used.value

    def submit(self, srv, nodes=(0,)):
        v, ticket = np.asarray(nodes, np.int32), ctypes.c_int64()
        assert self.lib.rs_server_submit(srv, 0, _ptr(v), ctypes.c_int64(v.size), None, None, ctypes.c_int64(0), 4,
                                         ctypes.byref(ticket)) == 0

    def poll(self, srv, block=1):
        tickets, status, path = np.zeros(8, np.int64), np.zeros(8, np.int32), np.zeros(8, np.int32)
        n = ctypes.c_int32()
        assert self.lib.rs_server_poll(srv, 8, 0, _ptr(tickets), _ptr(status), _ptr(path), None, None, ctypes.byref(n), block) == 0
        return list(zip(status[: n.value].tolist(), path[: n.value].tolist()))


@pytest.fixture
def calls(lib):
    lib.fake_fail_allocation(-1)
    return Calls(lib)


@pytest.mark.parametrize("hubs", [1, 3])
def test_hub_lists_are_ordered_before_their_readers(lib, calls, hubs):
    """A build, removals that find the lists long enough and keep them, a re-split of the rows and
    requests rescored on a server's copies: no kernel runs beside a copy that nothing orders
    before it."""
    lib.fake_classes(N - hubs, 0, 0, hubs, DEGREE, DEGREE, 3)
    before = lib.fake_launches(b"hub_p1_insert"), lib.fake_launches(b"hub_distinct")
    g = calls.build()
    assert calls.score(g) == 0
    for left in (hubs, max(1, hubs - 1)):
        lib.fake_classes(N - left, 0, 0, left, DEGREE, DEGREE, 3)
        assert calls.remove(g) == 0 and calls.score(g) == 0
    lib.fake_classes(N - hubs, 0, 0, hubs, DEGREE, DEGREE, 3)
    srv = calls.server([g], mode=1)
    for _ in range(2):
        calls.submit(srv)
        assert calls.poll(srv) == [(0, 0)]
    lib.rs_server_free(srv)
    after = lib.fake_launches(b"hub_p1_insert"), lib.fake_launches(b"hub_distinct")
    assert all(b - a >= 5 for a, b in zip(before, after))         # the paths with hub rows ran
    assert lib.fake_unordered() == b""


def test_every_failed_allocation_of_a_build(lib, calls):
    lib.fake_classes(N - 2, 0, 0, 2, DEGREE, DEGREE, 3)
    before = lib.fake_live_bytes()
    for n in range(200):
        lib.fake_fail_allocation(n)
        off, g = np.arange(N + 1) * DEGREE, ctypes.c_void_p()
        cols, labels = np.zeros(N * DEGREE, np.int32), np.zeros(N, np.int32)
        rc = lib.rs_build_graph(ctypes.c_int64(N), ctypes.c_int64(N * DEGREE), _ptr(off), 1, _ptr(cols), _ptr(labels), 8, 0, 0,
                                calls.s, ctypes.byref(g))
        if rc == 0:
            break
        assert rc == 2 and not g.value and lib.fake_live_bytes() == before, n          # RS_ENOMEM
    lib.fake_fail_allocation(-1)
    assert n > 40 and calls.score(g) == 0
    lib.rs_free_graph(g)
    assert lib.fake_live_bytes() == before


def test_a_graph_whose_change_failed_is_not_scored(lib, calls):
    """Removals that need longer hub lists and tables than there are, with each of the allocations
    failing: the scoring that follows is refused, not run on what is missing."""
    before = lib.fake_live_bytes()
    for n in range(40):
        lib.fake_classes(N, 0, 0, 0, 0, 0, 0)
        g = calls.build()
        lib.fake_classes(N - 3, 0, 0, 3, DEGREE, DEGREE, 3)
        lib.fake_fail_allocation(n)
        rc = calls.remove(g)
        lib.fake_fail_allocation(-1)
        ran = lib.fake_launches(b"hub_p1_insert")
        if rc == 0:
            break
        assert rc == 2 and calls.score(g) == 1 and lib.fake_launches(b"hub_p1_insert") == ran, n      # RS_ENOMEM, RS_EINVAL
        step = ctypes.c_void_p()
        assert lib.rs_step_capture(g, _ptr(calls.scores), 0, None, None, ctypes.byref(step)) == 1
        assert calls.remove(g) == 0 and calls.score(g) == 0 and lib.fake_launches(b"hub_p1_insert") == ran + 1
        lib.rs_free_graph(g)
        assert lib.fake_live_bytes() == before
    assert n > 8 and calls.score(g) == 0
    lib.rs_free_graph(g)


def test_a_failed_removal_writes_no_count(lib, calls):
    lib.fake_classes(N, 0, 0, 0, DEGREE, 0, 0)
    g, applied = calls.build(), ctypes.c_int64(-7)
    lib.fake_classes(N - 3, 0, 0, 3, DEGREE, DEGREE, 3)
    lib.fake_fail_allocation(0)
    assert calls.remove(g, applied=applied) == 2 and applied.value == -7
    lib.fake_fail_allocation(-1)
    assert calls.remove(g, applied=applied) == 0 and applied.value == 0     # (the stand-in's kernels count nothing)
    lib.rs_free_graph(g)


@pytest.mark.parametrize("n", [64, 30_000, 300_000])
def test_memory_of_slots_and_copies(lib, calls, n):
    """A slot takes 64 bytes a node beside its pools and a copy of a graph is counted as 170 a node and
    38 an entry: a budget that held so many slots and copies holds them, and the copy fits its share."""
    lib.fake_classes(n, 0, 0, 0, DEGREE, 0, 0)
    g, nnz = calls.build(n=n), n * DEGREE
    tcap, xcap = min(n, max(1 << 16, n // 4)), min(nnz, max(1 << 20, nnz // 4))
    # dead bits, flags, touched rows and their tables, W and scores, sums, pairs, triangles, lists, ranking
    slot = (nnz + 31) // 32 * 4 + 8 * n + 4 * tcap + 80 * tcap + 8 * (4 * xcap + 2 * tcap) + 8 * xcap + 64
    slot += 8 * n + 16 * n + 8 * n + 24 + 8 * xcap + 12 * xcap + 4 + 4 * (1 << 16) + 12 * 4 + (2 * n + 16384) * 12 + 64
    srv = calls.server([g], slots=2, budget=2 * slot, mode=1)
    slots = ctypes.c_int32()
    assert lib.rs_server_info(srv, ctypes.byref(slots), None, None, None) == 0
    assert slots.value == 2 and calls.used(srv) == 2 * slot
    lib.rs_server_free(srv)
    g, copy = calls.build(n=n), 38 * nnz + 170 * n + (16 << 20)
    srv = calls.server([g], slots=1, budget=slot + copy, mode=1)
    before = lib.fake_live_bytes()
    calls.submit(srv)
    assert calls.poll(srv) == [(0, 0)]
    assert calls.used(srv) == slot + copy and lib.fake_live_bytes() - before <= copy - (16 << 20)
    lib.rs_server_free(srv)


@pytest.mark.parametrize("n", [64, 10_000])
def test_memory_without_the_mirror_pass(lib, calls, n):
    lib.fake_classes(n, 0, 0, 0, DEGREE, 0, 0)
    g, nnz = calls.build(n=n), n * DEGREE
    calls.scores = np.zeros(n)
    tiles = 4 * (nnz // 2048 + 2)
    with_pass = lib.fake_live_bytes()
    for _ in range(2):
        assert calls.tune(g, p3_mirror=0) == 0 and lib.fake_live_bytes() == with_pass - 8 * nnz - tiles
        assert calls.score(g) == 0
        c = ctypes.c_void_p()
        before = lib.fake_live_bytes()
        lib.fake_classes(n - 2, 0, 0, 2, DEGREE, DEGREE, 3)      # (the hubs' scratch tables need more than 8 bytes a slot)
        assert lib.rs_clone_graph(g, ctypes.byref(c), calls.s) == 0 and calls.score(c) == 0
        lib.rs_free_graph(c)
        assert lib.fake_live_bytes() == before
        lib.fake_classes(n, 0, 0, 0, DEGREE, 0, 0)
        assert calls.tune(g, p3_mirror=1) == 0 and lib.fake_live_bytes() == with_pass
        assert calls.score(g) == 0
    lib.rs_free_graph(g)


@pytest.mark.parametrize("to", [0, 1])
def test_a_failed_change_of_the_mirror_pass(lib, calls, to):
    """Each allocation of the change failing: the setting before it stays, with its buffers."""
    lib.fake_classes(N, 0, 0, 0, DEGREE, 0, 0)
    g = calls.build()
    assert calls.tune(g, p3_mirror=1 - to) == 0
    held = lib.fake_live_bytes()
    for n in range(1 + to):
        lib.fake_fail_allocation(n)
        assert calls.tune(g, p3_mirror=to) == 2                     # RS_ENOMEM
        lib.fake_fail_allocation(-1)
        assert lib.fake_live_bytes() == held and calls.score(g) == 0
    assert calls.tune(g, p3_mirror=to) == 0 and calls.score(g) == 0
    lib.rs_free_graph(g)
