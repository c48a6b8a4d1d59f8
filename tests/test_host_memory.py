"""csrc/api.cu against a CUDA runtime made of host memory (fake_cuda.cpp): what the calls do when memory runs out, and
beside one another."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_cs_0408034_b200 import plogp

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
OUT = C.c_void_p(1 << 20)  # outputs are passed on to the kernels, which the fake ones leave alone


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fake") / "libplogp_fake.so")
    csrc = os.path.join(ROOT, "paper_cs_0408034_b200", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I/usr/local/cuda/include", "-x", "c++",
                    os.path.join(csrc, "api.cu"), os.path.join(ROOT, "tests", "fake_cuda.cpp"), "-o", so], check=True)
    lib = C.CDLL(so)
    lib.plogp_table_load.argtypes = [C.c_int, C.c_int, C.c_void_p, C.c_int, C.c_void_p, C.c_void_p, C.c_void_p]
    lib.plogp_select_best.argtypes = [C.c_void_p] * 6
    lib.plogp_predict.argtypes = [C.c_void_p] * 5
    lib.plogp_select_best_collective.argtypes = [C.c_void_p, C.c_void_p, C.c_int] + [C.c_void_p] * 4
    lib.plogp_table_free.argtypes = [C.c_void_p]
    lib.plogp_select_best_host.argtypes = [C.c_void_p] * 6
    lib.plogp_segment_surface.argtypes = [C.c_void_p] * 4
    lib.plogp_profile_read.argtypes = [C.c_void_p] * 3
    lib.fake_refuse_from.argtypes = lib.fake_refuse_host_from.argtypes = [C.c_longlong]
    for f in ("fake_bad_accesses", "fake_launches", "fake_live_bytes", "fake_too_large", "fake_staged", "fake_direct"):
        getattr(lib, f).restype = C.c_longlong
    return lib


def load(lib, n_tables, n_bp=3):
    sizes = np.array([4, 1024, 1 << 20], dtype=np.uint64) if n_bp == 3 else 4 * np.arange(1, n_bp + 1, dtype=np.uint64)
    gaps = np.ascontiguousarray(np.tile([1.0, 2.0, 900.0] if n_bp == 3 else np.arange(1.0, n_bp + 1), (n_tables, 1)))
    h = C.c_void_p()
    lat = np.full(n_tables, 5.0)
    assert lib.plogp_table_load(n_tables, n_bp, sizes.ctypes.data, 1, gaps.ctypes.data, lat.ctypes.data, C.byref(h)) == plogp.OK
    return h


def long_list(P_hi, n_m, **kw):
    return plogp.GridArgs(np.arange(1, n_m + 1) * 65536, None, 2, P_hi, None, s_lo=4, s_hi=4096, s_step=4, **kw)


@pytest.mark.parametrize("kind", ["sweep", "envelope", "gaps", "predict"])
def test_scratch_that_does_not_grow_leaves_no_call_without_it(lib, kind):
    """A grid whose scratch is refused: its call says so, and a call on a grid that the handle has kept a plan for either
    gets scratch of its own or says so too, before any kernel is launched."""
    short = plogp.GridArgs(np.arange(1, 129) * 4096, None, 2, 700, np.array([64, 256, 1024, 4096]))
    small = short if kind in ("gaps", "predict") else long_list(40, 3, search_mode=int(kind == "envelope"))
    large = long_list(3000, 60)
    h = load(lib, 300)

    def call():
        if kind == "predict":
            return lib.plogp_predict(h, small.ref, OUT, None, None)
        return lib.plogp_select_best(h, small.ref, OUT, OUT, OUT, None)

    try:
        assert call() == plogp.OK
        for refused_too in (False, True):
            lib.fake_refuse_from((64 << 10) if refused_too else (64 << 20))
            assert lib.plogp_select_best(h, large.ref, OUT, OUT, OUT, None) == plogp.E_NOMEM
            n = lib.fake_launches()
            assert call() == (plogp.E_NOMEM if refused_too else plogp.OK)
            assert lib.fake_bad_accesses() == 0 and (lib.fake_launches() == n) == refused_too
            lib.fake_refuse_from(-1)
            assert call() == plogp.OK and lib.fake_bad_accesses() == 0
        assert lib.plogp_select_best(h, large.ref, OUT, OUT, OUT, None) == plogp.OK and lib.fake_bad_accesses() == 0
    finally:
        lib.fake_refuse_from(-1)
        lib.plogp_table_free(h)
    assert lib.fake_live_bytes() == 0


@pytest.mark.parametrize("mine,theirs", [(100 << 10, 60 << 10), (60 << 10, 100 << 10), (227 << 10, 49 << 10), (100 << 10, 1 << 10)])
def test_launches_of_one_kernel_from_two_threads(lib, mine, theirs):
    """Handles are independent: a call that needs less shared memory does not lower a kernel's limit for one on another thread
    that has just raised it."""
    assert lib.fake_launch_beside(mine, theirs)


def in_a_child(f):
    """Exit status of f() in a process of its own: an exception that leaves a C call ends it with a signal."""
    pid = os.fork()
    if pid == 0:
        os._exit(0 if f() else 1)
    return os.waitpid(pid, 0)[1]


@pytest.mark.parametrize("refuse", [1, 64, 600, 5000])
def test_host_memory_that_runs_out_is_a_status(lib, refuse):
    """Allocations of a size and up fail while a plan is built: every call returns PLOGP_E_NOMEM (or succeeds), nothing throws,
    and the calls go on afterwards."""
    grids = [long_list(300, 40), long_list(300, 40, search_mode=1), plogp.GridArgs(np.arange(1, 101) * 4096, None, 2, 700, np.arange(4, 100, 4))]

    def f():
        h = load(lib, 8)
        kept = long_list(20, 2)
        ok = lib.plogp_select_best(h, kept.ref, OUT, OUT, OUT, None) == plogp.OK
        for g in grids:
            calls = [lambda: lib.plogp_select_best(h, g.ref, OUT, OUT, OUT, None), lambda: lib.plogp_predict(h, g.ref, OUT, None, None),
                     lambda: lib.plogp_select_best_collective(h, g.ref, 4, OUT, OUT, OUT, None), lambda: lib.plogp_segment_surface(h, g.ref, OUT, None)]
            for call in calls:
                lib.fake_refuse_host_from(refuse)
                ok &= call() in (plogp.OK, plogp.E_NOMEM)
                if refuse == 1:
                    ok &= lib.plogp_select_best(h, kept.ref, OUT, OUT, OUT, None) in (plogp.OK, plogp.E_NOMEM)
                lib.fake_refuse_host_from(-1)
                ok &= call() == plogp.OK and lib.plogp_select_best(h, kept.ref, OUT, OUT, OUT, None) == plogp.OK
        lib.plogp_profile_enable(C.c_void_p(h.value), 1)
        lib.fake_refuse_host_from(refuse)
        ok &= all(lib.plogp_select_best(h, kept.ref, OUT, OUT, OUT, None) == plogp.OK for _ in range(300))
        return ok & (lib.plogp_table_free(h) == plogp.OK) & (lib.fake_live_bytes() == 0) & (lib.fake_bad_accesses() == 0)

    assert in_a_child(f) == 0


def test_device_memory_that_runs_out_for_a_grid_is_a_status(lib):
    g, h = long_list(300, 40), load(lib, 8)
    lib.fake_refuse_from(1)
    assert lib.plogp_select_best(h, g.ref, OUT, OUT, OUT, None) == plogp.E_NOMEM
    lib.fake_refuse_from(-1)
    assert lib.plogp_select_best(h, g.ref, OUT, OUT, OUT, None) == plogp.OK
    assert lib.plogp_table_free(h) == plogp.OK


def octaves(n):
    """256 and more listed process counts over n octaves, two (floor, ceil) pairs of log2 P in each."""
    return np.unique(np.concatenate([1 << np.arange(1, n), np.rint(2.0 ** np.linspace(1.5, n - 0.5, 256))])).astype(np.int32)


@pytest.mark.parametrize("n_bp", [64, 1024])
@pytest.mark.parametrize("n_m,P,n_s,n_tables", [
    (255, 512, 64, 1200), (253, 1024, 24, 900), (255, 3000, 32, 900), (250, 512, 32, 900), (255, 512, 24, 900), (255, 29, 24, 900), (255, 29, 32, 600), (229, 29, 8, 900),
    (201, 29, 32, 900), (173, 29, 20, 900), (157, 29, 64, 900), (256, 29, 64, 900), (127, 512, 32, 900), (33, 29, 64, 900), (19, 29, 7, 1), (1, 29, 64, 1)])
def test_shared_memory_fits(lib, n_m, P, n_s, n_tables, n_bp):
    """Every launch on a short candidate list has at most the shared memory of an SM, whatever the message sizes, the candidates
    and the (floor, ceil) pairs of log2 P are: P = 2..P, or listed over P octaves."""
    listed = octaves(P) if P < 30 else None
    grid = plogp.GridArgs(np.arange(1, n_m + 1) * 64, listed, 2, P, np.arange(1, n_s + 1) * 8)
    h = load(lib, n_tables, n_bp)
    try:
        for call in (lambda: lib.plogp_select_best(h, grid.ref, OUT, OUT, OUT, None), lambda: lib.plogp_predict(h, grid.ref, OUT, OUT, None),
                     lambda: lib.plogp_select_best_collective(h, grid.ref, 3, OUT, OUT, OUT, None)):
            n = lib.fake_too_large()
            assert call() == plogp.OK and lib.fake_too_large() == n and lib.fake_bad_accesses() == 0
    finally:
        lib.plogp_table_free(h)


def test_scratch_of_very_long_lists(lib):
    """Two thousand million candidates, 65535 process counts: partial minima of 32 chunks per message size, 3.2 GB, and not of
    chunks as short as they are elsewhere."""
    n_m = 64
    grid = plogp.GridArgs((1 << 31) + np.arange(n_m), None, 2, 65536, None, s_lo=1, s_hi=(1 << 31) - 1, s_step=1, dtype_bytes=1, strategy_mask=0x24)
    h = load(lib, 1)
    try:
        lib.fake_refuse_from(n_m * 33 * 2 * 65535 * 12)
        assert lib.plogp_select_best(h, grid.ref, OUT, OUT, OUT, None) == plogp.OK and lib.fake_bad_accesses() == 0
    finally:
        lib.fake_refuse_from(-1)
        lib.plogp_table_free(h)


@pytest.mark.parametrize("n_tables,n_P,n_m,n_s,cells", [(1, 49, 19, 7, True), (3, 74, 8, 43, True), (500, 29, 8, 5, True), (1, 1023, 256, 64, False), (64, 511, 128, 32, False),
                                                        (2, 70, 19, 8, True), (900, 70, 19, 8, False), (900, 30, 33, 64, False)])
def test_which_grids_have_a_cell_per_thread(lib, n_tables, n_P, n_m, n_s, cells):
    grid = plogp.GridArgs(np.arange(1, n_m + 1) * 4096, None, 2, n_P + 1, np.arange(1, n_s + 1) * 64)
    h = load(lib, n_tables)
    try:
        for call in (lambda: lib.plogp_select_best(h, grid.ref, OUT, OUT, OUT, None), lambda: lib.plogp_predict(h, grid.ref, OUT, OUT, None)):
            n = lib.fake_direct()
            assert call() == plogp.OK and lib.fake_direct() - n == cells and lib.fake_bad_accesses() == 0
    finally:
        lib.plogp_table_free(h)


@pytest.mark.parametrize("n_tables,n_P,n_m,n_s,launches", [(1, 49, 19, 7, 1), (1, 1023, 256, 64, 1), (4, 2696, 33, 14, 1), (200, 99, 9, 10, 1), (9, 668, 19, 7, 1), (48, 1384, 24, 10, 1), (60, 1805, 8, 33, 2),
                                                           (17, 201, 185, 8, 1), (64, 511, 128, 32, 2), (4096, 511, 128, 32, 3)])
def test_launches_of_a_decision(lib, n_tables, n_P, n_m, n_s, launches):
    """One where both halves have room beside one another; the gap pre-pass on large grids."""
    grid = plogp.GridArgs(np.arange(1, n_m + 1) * 4096, None, 2, n_P + 1, np.arange(1, n_s + 1) * 64)
    h = load(lib, n_tables)
    try:
        n = lib.fake_launches()
        assert lib.plogp_select_best(h, grid.ref, OUT, OUT, OUT, None) == plogp.OK and lib.fake_launches() - n == launches
    finally:
        lib.plogp_table_free(h)


@pytest.mark.parametrize("n_tables,n_P,n_m,n_s,decide,predict", [
    (900, 257, 127, 24, 1, 1), (900, 97, 33, 33, 1, 0), (900, 256, 201, 3, 1, 1), (450, 520, 99, 9, 1, 1), (600, 193, 34, 20, 0, 1), (600, 257, 52, 32, 0, 1),
    (600, 260, 250, 32, 0, 1), (600, 256, 255, 20, 0, 1), (900, 257, 65, 24, 0, 1), (900, 97, 127, 24, 0, 1), (900, 95, 33, 33, 0, 0), (900, 31, 145, 9, 1, 1), (900, 28, 195, 29, 1, 0),
    (900, 14, 65, 40, 1, 1), (900, 172, 195, 8, 0, 1), (900, 50, 99, 8, 0, 0),
    (900, 1100, 127, 32, 1, 1), (900, 257, 127, 64, 0, 0), (300, 257, 127, 24, 0, 0), (900, 257, 128, 24, 0, 0), (900, 257, 31, 8, 0, 0), (900, 257, 257, 8, 0, 0)])
def test_which_grids_have_all_message_sizes_in_a_cta(lib, n_tables, n_P, n_m, n_s, decide, predict):
    grid = plogp.GridArgs(np.arange(1, n_m + 1) * 4096, None, 2, n_P + 1, np.arange(1, n_s + 1) * 64)
    h = load(lib, n_tables, 64)
    try:
        for out, want in ((OUT, (decide, predict)), (C.c_void_p(OUT.value + 8), (0, 0))):
            for call, n in zip((lambda: lib.plogp_select_best(h, grid.ref, out, out, out, None), lambda: lib.plogp_predict(h, grid.ref, out, out, None)), want):
                before = lib.fake_staged()
                assert call() == plogp.OK and lib.fake_staged() - before == n and lib.fake_too_large() == 0
    finally:
        lib.plogp_table_free(h)
