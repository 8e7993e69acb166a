"""The checked build flavour of the library (``libtsenor_bounds.so``: the same sources compiled with
-DTSENOR_BOUNDS, every computed index of the loaders, the rounding tables, the local search and the
writers tested before use, a bad one reported as TSENOR_DEV_INTERNAL and skipped).  It stands in for
a memory checker: on every block size, both fixed register layouts and the builds that only the automatic
choice reaches, wide matrices with a ragged last unit and slabs, no index check may fire, and the results
must equal the normal library's."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2505_23949_b200 import binding as ts
from paper_2505_23949_b200 import build as ts_build
from paper_2505_23949_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

SHAPES = [(4, 2, 8, 516), (8, 3, 16, 520), (16, 8, 32, 272), (32, 16, 64, 160), (32, 7, 32, 32),
          (4, 2, 4 * 259, 4), (8, 4, 8 * 131, 8), (16, 8, 16 * 35, 16), (32, 16, 32 * 11, 32)]


@pytest.fixture()
def checked_library():
    """Swaps the binding's library for the checked flavour for the duration of a test."""
    path = ts_build.build(bounds=True)
    normal_path, normal_lib = ts.LIB_PATH, ts.lib()
    ts._lib, ts.LIB_PATH = None, path
    try:
        assert ts.lib() is not normal_lib
        yield
    finally:
        ts._lib, ts.LIB_PATH = normal_lib, normal_path


def _run_all(M, N, rows, cols, layout, iters=60):
    ts.set_layout(layout)
    W = synth.student_t_abs(rows, cols, 0.02, seed=31 * M + N)
    Wd = torch.from_numpy(W).to(DEV)
    tau = synth.default_tau(float(W.max()))
    st = ts.new_status(DEV)
    mask = ts.solve(Wd, N, M, tau, iters, -1, status=st)
    plan = ts.dykstra(Wd, N, M, tau, iters, plan_is_log=True, status=st)
    strict = ts.round_plan(plan, Wd, N, M, ls_steps=1, status=st)
    ee = ts.solve_scores(ts.Scores(ts.SCORES_ABS, Wd, early_exit_eps=1e-2), N, M, tau, iters, -1, status=st)
    torch.cuda.synchronize()
    ts.set_layout(ts.LAYOUT_AUTO)
    return int(st.item()), [t.cpu().numpy() for t in (mask, plan, strict, ee)]


@pytest.mark.parametrize("layout", [ts.LAYOUT_THROUGHPUT, ts.LAYOUT_LATENCY])
@pytest.mark.parametrize("M,N,rows,cols", SHAPES)
def test_no_index_check_fires_and_results_equal_the_normal_build(checked_library, M, N, rows, cols, layout):
    flags, got = _run_all(M, N, rows, cols, layout)
    assert (flags & ts.DEV_INTERNAL) == 0, "an index check fired"
    checked, checked_path = ts._lib, ts.LIB_PATH
    ts._lib, ts.LIB_PATH = None, ts_build.LIB
    try:
        flags_n, want = _run_all(M, N, rows, cols, layout)
    finally:
        ts._lib, ts.LIB_PATH = checked, checked_path
    assert flags == flags_n
    for g, w in zip(got, want):
        assert np.array_equal(g, w)


# sizes whose builds only the automatic choice reaches: spread (M = 8, 16)
@pytest.mark.parametrize("M,N,rows,cols", [(8, 3, 768, 776), (16, 5, 640, 656), (16, 8, 1040, 1008)])
def test_no_index_check_fires_under_the_automatic_choice(checked_library, M, N, rows, cols):
    iters = 60 if rows < 1000 else 300
    flags, got = _run_all(M, N, rows, cols, ts.LAYOUT_AUTO, iters)
    assert (flags & ts.DEV_INTERNAL) == 0 and _checks_that_fired() == 0
    checked, checked_path = ts._lib, ts.LIB_PATH
    ts._lib, ts.LIB_PATH = None, ts_build.LIB
    try:
        flags_n, want = _run_all(M, N, rows, cols, ts.LAYOUT_AUTO, iters)
    finally:
        ts._lib, ts.LIB_PATH = checked, checked_path
    assert flags == flags_n
    for g, w in zip(got, want):
        assert np.array_equal(g, w)


def _checks_that_fired():
    """What the checked flavour keeps for entry points without a status word."""
    seen = torch.full((1,), -1, dtype=torch.int32, device=DEV)
    assert ts.lib().tsenor_bounds_seen(ctypes.c_void_p(seen.data_ptr()), ts._stream(None)) == ts.OK
    return int(seen.item())


# slabs, ragged widths, padded mask words, and numbers of units that do not fill a CTA's four warps
@pytest.mark.parametrize("M,N,rows,cols", SHAPES + [(4, 1, 4, 4), (8, 3, 8 * 5, 8 * 9), (16, 5, 16 * 3, 16 * 3),
                                                    (32, 9, 32 * 3, 32 * 7), (32, 1, 32, 32)])
def test_simple_rounding_under_the_checked_flavour(checked_library, M, N, rows, cols):
    key = torch.from_numpy(synth.student_t_abs(rows, cols, 1.0, seed=M + N)).to(DEV)
    got = ts.simple_round(key, N, M, mask_out=ts.new_mask(rows, cols, DEV).fill_(-1)).cpu().numpy().view(np.uint32)
    assert _checks_that_fired() == 0
    assert np.array_equal(got, oracle.simple_round(key.cpu().numpy(), N, M))
