"""Tasks of the front sweeps. Where a kernel streams a task's input rows past its
four warps, a task must hold at most one group of 16 output rows per warp: the
rows pass once, in windows of two buffers, and a warp's second group would read
rows that have already gone. The persistent form (persistent_sweeps = 1)
streams every task; the per-level form streams the levels whose longest
reduction does not fit in shared memory."""
import ctypes as C
import os

import numpy as np
import pytest

from paper_2004_07930_gb300 import build as hzbuild
from paper_2004_07930_gb300 import hz
from paper_2004_07930_gb300 import workloads as wl

from _gpu_common import torch_cuda

WARPS, GROUP, RESIDENT = 4, 16, 256


@pytest.fixture(scope="module")
def lib():
    if not os.path.exists(hzbuild.LIB):
        hzbuild.build()
    L = hz.load()
    I = C.POINTER(C.c_int)
    L.hz_internal_level_tasks.argtypes = [C.c_int, C.c_int, C.c_int, C.c_int, I, I, I, C.c_int, I]
    return L


def level_tasks(lib, fwd, fp32, stream, k, f):
    I = C.POINTER(C.c_int)
    k, f = np.ascontiguousarray(k, np.int32), np.ascontiguousarray(f, np.int32)
    out = np.zeros((int(((f + GROUP - 1) // GROUP).sum()), 3), np.int32)
    rows = C.c_int()
    n = lib.hz_internal_level_tasks(fwd, fp32, stream, len(k), k.ctypes.data_as(I), f.ctypes.data_as(I),
                                    out.ctypes.data_as(I), len(out), C.byref(rows))
    assert n <= len(out)
    return out[:n], rows.value


def streamed_reads_in_window(fwd, k, f, g0, ng, window):
    """Every reduction index that a warp's groups read lies in the window of
    input rows that is in shared memory when they read it."""
    lo, hi = (0, min(k, GROUP * (g0 + ng))) if fwd else (GROUP * g0, f)
    for warp in range(WARPS):
        base = lo
        for g in range(g0 + warp, g0 + ng, WARPS):
            first, last = (0, min(k, GROUP * (g + 1))) if fwd else (GROUP * g, f)
            if first < last and first < base:
                return False
            while base + window < min(last, hi):
                base += window
    return True


# (fronts, pivots, order) of one level: many small fronts (tasks of up to 16 groups where the inputs are
# staged whole), more pivots than a window, one front only, a reduction that does not fit
LEVELS = [(2000, 62, 208), (800, 100, 240), (5000, 30, 250), (1, 256, 256), (3, 40, 41), (900, 60, 300), (40, 500, 1400)]


@pytest.mark.parametrize("fp32", [1, 0])
@pytest.mark.parametrize("fwd", [1, 0])
@pytest.mark.parametrize("count,k,f", LEVELS)
def test_streamed_tasks_read_rows_that_are_there(lib, fwd, fp32, count, k, f):
    kk, ff = np.full(count, k), np.full(count, f)
    for stream in (1, 0):
        tasks, rows = level_tasks(lib, fwd, fp32, stream, kk, ff)
        assert rows == (k if fwd else f)
        nout = f if fwd else k
        cover = np.zeros((count, (nout + GROUP - 1) // GROUP), int)
        for front, g0, ng in tasks:
            cover[front, g0:g0 + ng] += 1
        assert (cover == 1).all()
        if stream or rows > RESIDENT:
            assert tasks[:, 2].max() <= WARPS
            for front, g0, ng in tasks[:64]:
                for window in (32, 64, 128):
                    assert streamed_reads_in_window(fwd, k, f, int(g0), int(ng), window)


def test_tasks_of_large_levels_stay_wide_where_they_are_staged_whole(lib):
    """The per-level form keeps its tasks of many groups (which the streamed
    form could not run)."""
    tasks, rows = level_tasks(lib, 1, 1, 0, np.full(2000, 62), np.full(2000, 208))
    assert rows <= RESIDENT and tasks[:, 2].max() > WARPS
    assert not streamed_reads_in_window(1, 62, 208, 0, int(tasks[:, 2].max()), 32)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [hz.HZ_PREC_FP64, hz.HZ_PREC_MIXED])
def test_persistent_equals_per_level_on_wide_tasks(precision):
    """A problem whose per-level tasks have more groups than warps, with more
    pivots than a window of input rows: the two forms agree bit for bit."""
    torch_cuda()
    p = wl.cube_problem(ncell=16, nparts_xyz=(2, 2, 2), coarse=False)
    opts = dict(precision=precision, coarse_mode=hz.HZ_COARSE_NONE)
    with hz.Solver.from_problem(p, persistent_sweeps=1, **opts) as Sp, \
            hz.Solver.from_problem(p, persistent_sweeps=0, **opts) as Sl:
        groups = Sp._lib.hz_internal_task_groups
        groups.argtypes = [C.c_void_p]
        assert groups(Sl._ctx) > WARPS and groups(Sp._ctx) <= WARPS
        for s in (1, 3, 16):
            X = wl.random_rhs(Sp.n, s, 50 + s)
            Yp = Sp.apply_prec(X)
            assert np.isfinite(Yp).all()
            np.testing.assert_array_equal(Yp, Sp.apply_prec(X))
            np.testing.assert_array_equal(Yp, Sl.apply_prec(X))
