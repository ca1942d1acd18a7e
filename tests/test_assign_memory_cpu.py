"""The assignment engine's device memory, without a GPU: the library's host code
linked against a CUDA runtime that only keeps account of allocations, copies
and launches (fake_cudart.cpp; no kernel runs)."""
from __future__ import annotations

import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
P = ctypes.c_void_p
E_OOM = -2


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2406_08496_gb300 import _build
    out = tmp_path_factory.mktemp("fake")
    objs = []
    # (the fake first: its tables are there before the kernels register)
    for src in (os.path.join(HERE, "fake_cudart.cpp"), os.path.join(_build.CSRC, "assign.cpp"),
                os.path.join(_build.CSRC, "assign_gpu.cu")):
        objs.append(str(out / (os.path.basename(src) + ".o")))
        r = subprocess.run([_build._nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, "-Xptxas", "-v", "-c", src, "-o", objs[-1]],
                           check=True, capture_output=True, text=True)
    so = str(out / "libfake.so")
    subprocess.run(["g++", "-shared", "-o", so, *objs, "-lpthread"], check=True)
    report = r.stderr  # of assign_gpu.cu, the last
    lib = ctypes.CDLL(so, mode=os.RTLD_LOCAL | os.RTLD_NOW | os.RTLD_DEEPBIND)
    u32, u64 = ctypes.c_uint32, ctypes.c_uint64
    lib.lpsim_assign_create.argtypes = [P, u32, u32, P, P, P, P, P, u64, P, P, P, P, P, ctypes.c_float, u64]
    lib.lpsim_assign_shortest_paths_gpu.argtypes = [P, P, u32, u32, u32, P]
    lib.lpsim_assign_load_gpu.argtypes = [P, P, u32, u32, P]
    lib.lpsim_assign_destroy.argtypes = [P]
    lib.lpsim_assign_shortest_paths.argtypes = [P, P, u32, u32, u32, u32, P]
    lib.lpsim_assign_reroute.argtypes = [P, ctypes.c_double, u32, P]
    lib.fake_reset.argtypes = [ctypes.c_long]
    lib.fake_next_read.argtypes = [ctypes.c_size_t, u64]
    lib.fake_launch.argtypes = [ctypes.c_int, P]
    lib.fake_launch.restype = ctypes.c_char_p
    lib.fake_occupancy.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_size_t]
    for f in ("fake_calls", "fake_uploaded", "fake_live_bytes"):
        getattr(lib, f).restype = ctypes.c_long
    lib.compiler_report = report
    return lib


def _p(a):
    return a.ctypes.data_as(P)


class _Engine:
    """A ring of nodes, both ways round, and trips from a few of them."""

    def __init__(self, lib, n_nodes, n_trips=64, origins=4, hops=2):
        self.lib, self.n = lib, n_trips
        i = np.arange(n_nodes, dtype=np.uint32)
        src, dst = np.concatenate([i, i]), np.concatenate([(i + 1) % n_nodes, (i + n_nodes - 1) % n_nodes]).astype(np.uint32)
        self.m = len(src)
        length, lanes, vmax = np.full(self.m, 100.0, np.float32), np.ones(self.m, np.uint8), np.full(self.m, 10.0, np.float32)
        orig = (np.arange(n_trips) % origins).astype(np.uint32)
        dest, dep = ((orig + hops) % n_nodes).astype(np.uint32), np.arange(n_trips, dtype=np.uint32)
        off = hops * np.arange(n_trips + 1, dtype=np.uint64)
        edges = ((orig[:, None] + np.arange(hops)) % n_nodes).reshape(-1).astype(np.uint32)
        h = P()
        self._keep = (src, dst, length, lanes, vmax, orig, dest, dep, off, edges)
        assert lib.lpsim_assign_create(ctypes.byref(h), n_nodes, self.m, *[_p(a) for a in self._keep[:5]], n_trips,
                                       *[_p(a) for a in self._keep[5:]], 0.5, 1) == 0
        self.h = h

    def search(self, period, n_bins=4):
        tt, t = np.full((self.m, n_bins), 5.0, np.float32), np.empty(self.n, np.float32)
        return self.lib.lpsim_assign_shortest_paths_gpu(self.h, _p(tt), n_bins, 60, period, _p(t))

    def load(self, n_bins):
        tt, f = np.full((self.m, n_bins), 5.0, np.float32), np.empty((self.m, n_bins), np.uint32)
        return self.lib.lpsim_assign_load_gpu(self.h, _p(tt), n_bins, 60, _p(f))

    def close(self):
        self.lib.lpsim_assign_destroy(self.h)


def _launches(lib, first=0):
    out = []
    for i in range(first, lib.fake_launches()):
        v = np.empty(5, np.int32)
        name = lib.fake_launch(i, _p(v)).decode()
        out.append((name, *[int(x) for x in v]))
    return out


def _calls(lib, e):
    """Every kind of device allocation: set-up, a first search, another period, a
    path buffer that was too small, a loading, larger tables for both."""
    def too_small():
        lib.fake_next_read(8, 3 << 20)  # path edges asked for
        lib.fake_next_read(4, 2)        # the search's word: the path buffer was too small
        return e.search(7)
    return [lambda: e.search(600), lambda: e.search(7), too_small, lambda: e.load(4), lambda: e.load(8),
            lambda: e.search(600, 8)]


@pytest.mark.parametrize("n_nodes", [100, 60000])  # labels in shared memory; workspaces in device memory
def test_an_engine_survives_each_failed_allocation(lib, n_nodes):
    """One device allocation fails, each in turn: that call reports
    LPSIM_E_OOM, and every call after it allocates what is missing again, so
    that no kernel is launched on a freed or missing buffer."""
    before = lib.fake_live_bytes()
    e = _Engine(lib, n_nodes)
    lib.fake_reset(0)
    want = []  # launches of each call when nothing fails
    for call in _calls(lib, e):
        at = lib.fake_launches()
        assert call() == 0, lib.lpsim_last_error()
        want.append({(x[0], x[3]) for x in _launches(lib, at)})
    total = lib.fake_calls()
    e.close()
    assert lib.fake_live_bytes() == before and total > 20
    for n in range(1, total + 1):
        e = _Engine(lib, n_nodes)
        lib.fake_reset(n)
        rcs = []
        for call in _calls(lib, e):
            rcs.append(call())
        assert rcs.count(E_OOM) == 1 and rcs.count(0) == len(rcs) - 1, (n, rcs)
        for q, call in enumerate(_calls(lib, e)):
            at = lib.fake_launches()
            assert call() == 0, (n, q)
            for x in _launches(lib, at):
                assert (x[0], x[3]) in want[q] and x[4] == 0, (n, q, x, want[q])
        for x in _launches(lib):
            assert x[4] == 0, (n, x)
        e.close()
        assert lib.fake_live_bytes() == before


def test_search_of_large_networks_keeps_to_its_registers(lib):
    """td_trees runs 40 warps on an SM, which leaves 48 registers a thread: the
    compiler's report has it use no more and spill none."""
    at = lib.compiler_report.index("8td_trees")
    props = lib.compiler_report[at:].split("Used", 1)
    assert " 0 bytes spill stores, 0 bytes spill loads" in props[0], props[0]
    assert int(props[1].split()[0]) <= 48


@pytest.mark.parametrize("n_trips,origins,period", [(64, 4, 600), (3000, 600, 1)])
def test_a_small_engine_takes_little_device_memory(lib, n_trips, origins, period):
    """600 nodes: a loading needs no search workspace, a search of four trees one
    for four blocks, and a search of thousands no more than the warps' workspaces
    of a search in device memory (32 bytes per node for 40 trees on each of 152
    SMs), besides tables and a path buffer of some 5 MB."""
    before = lib.fake_live_bytes()
    e = _Engine(lib, 600, n_trips, origins)
    lib.fake_reset(0)
    assert e.load(4) == 0
    assert lib.fake_live_bytes() - before < 2 << 20
    assert e.search(period) == 0
    trees = len(set(zip((np.arange(n_trips) % origins).tolist(), (np.arange(n_trips) // period).tolist())))
    assert lib.fake_live_bytes() - before < (8 << 20) + (32 * 600 * 40 * 152 if trees > 4 else 4 << 20)
    e.close()
    assert lib.fake_live_bytes() == before


@pytest.mark.parametrize("n_nodes", [200, 6200, 6400, 8600, 10500, 10600, 13300, 13400, 18000, 18200, 20480, 27500, 27530,
                                     27640, 27700, 40000, 55800])
def test_the_search_s_block_follows_the_occupancy(lib, n_nodes):
    """The block a search launches is the one of which most fit an SM beside its
    tree's labels, and among those the one with most threads, then with most
    registers: no size runs fewer trees, or fewer threads per tree, than it could."""
    e = _Engine(lib, n_nodes)
    lib.fake_reset(0)
    assert e.search(600) == 0
    name, threads, _, _, _, smem = next(x for x in _launches(lib) if "td_trees" in x[0])
    assert "td_trees_shared" in name
    key = lambda t, r: (lib.fake_occupancy(t, r, smem), t, r)
    assert key(threads, 32 if "Li8E" in name else 56) == max(key(256, 32), key(256, 56), key(512, 56), key(1024, 56))
    e.close()


def test_a_small_rerouting_brings_little_to_the_device(lib):
    """4,000 trips of 60 edges on a ring, one in a hundred moved to the 40 edges
    the other way round: the next loading takes the moved routes and where each
    trip's route stands (16 bytes) to the device, not the routes that stay."""
    e = _Engine(lib, 100, 4000, 4, hops=60)
    tt, t = np.full((e.m, 4), 5.0, np.float32), np.empty(e.n, np.float32)
    assert lib.lpsim_assign_shortest_paths(e.h, _p(tt), 4, 60, 600, 2, _p(t)) == 0
    lib.fake_reset(0)
    assert e.load(4) == 0 and lib.fake_uploaded() > 4 * 60 * e.n
    at, changed = lib.fake_uploaded(), ctypes.c_uint64()
    assert lib.lpsim_assign_reroute(e.h, 0.01, 1, ctypes.byref(changed)) == 0 and 10 < changed.value < 100
    assert e.load(4) == 0
    assert lib.fake_uploaded() - at == tt.nbytes + 16 * e.n + 4 * 40 * changed.value
    assert e.load(4) == 0
    assert lib.fake_uploaded() - at == 2 * tt.nbytes + 16 * e.n + 4 * 40 * changed.value
    e.close()


def test_a_rewrite_leaves_room_for_the_next_small_rerouting(lib):
    """Routes that have grown by a fifth since the buffers were made (one trip in
    twenty on 60 edges instead of 10): small re-routings to and fro after that
    bring what they move, but for a few rewrites."""
    e = _Engine(lib, 70, 4000, 4, hops=10)
    tt, t, changed = np.full((e.m, 4), 5.0, np.float32), np.empty(e.n, np.float32), ctypes.c_uint64()
    lib.fake_reset(0)
    rewrites = 0
    for it, f in enumerate([0.045] + 40 * [0.004, 0.05]):
        back = it % 2 == 0  # the way back is 60 edges long, the way forward 10
        tt[:70], tt[70:] = (500.0, 5.0) if back else (5.0, 500.0)
        assert lib.lpsim_assign_shortest_paths(e.h, _p(tt), 4, 60, 600, 2, _p(t)) == 0
        assert lib.lpsim_assign_reroute(e.h, f if back else 0.1, it, ctypes.byref(changed)) == 0
        at = lib.fake_uploaded()
        assert e.load(4) == 0
        rewrites += lib.fake_uploaded() - at - tt.nbytes - 16 * e.n != 4 * (60 if back else 10) * changed.value
    assert rewrites <= 18  # of 81; 24 with buffers that only just hold the routes
    e.close()
