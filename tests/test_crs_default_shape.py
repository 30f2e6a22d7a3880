"""Default VECTOR shape of a CRS handle: lanes and rows at the limits of the
mean row length, in both types, and what a request for lanes alone makes of
the default's rows.  Host logic: handles over placeholder addresses."""
import ctypes

import pytest

from paper_0910_4836_gb300 import _lib

P = ctypes.c_void_p(256)  # never dereferenced on the host


def _handle(mean, dtype):
    h = ctypes.c_void_p()
    nnz = 64 * mean
    assert _lib.load().gbsp_crs_create(64, 64, nnz, P, P, P, dtype, ctypes.byref(h)) == 0
    return h


def _set(h, kernel, lanes=0, rows=0):
    o = _lib.KernelOpts(_lib.KERNELS[kernel], lanes, rows, 0, 0, 0)
    assert _lib.load().gbsp_set_kernel(h, ctypes.byref(o)) == 0


def _shape(h):
    o = _lib.KernelOpts()
    assert _lib.load().gbsp_get_kernel(h, ctypes.byref(o)) == 0
    return o.lanes, o.rows_per_warp


@pytest.mark.parametrize("mean,f64,f32", [
    (0, (1, 1), (1, 1)), (5, (1, 1), (1, 1)), (6, (2, 4), (2, 4)), (12, (4, 4), (4, 4)), (19, (4, 4), (4, 4)),
    (20, (4, 4), (8, 4)), (23, (4, 4), (8, 4)), (24, (4, 2), (8, 4)), (35, (4, 2), (8, 4)), (36, (8, 4), (8, 4)),
    (64, (16, 4), (16, 4)), (192, (32, 4), (32, 4))])
def test_default_shape(mean, f64, f32):
    for dtype, want in ((0, f64), (1, f32)):
        h = _handle(mean, dtype)
        try:
            assert _shape(h) == want
            for lanes in (1, 2, 8, 16, 4):  # the default's rows follow the lanes
                _set(h, "vector", lanes)
                assert _shape(h) == (lanes, 1 if lanes == 1 else 4)
            _set(h, "vector", 4, 2)         # rows that were asked for stay
            _set(h, "vector", 16)
            assert _shape(h) == (16, 2)
            _set(h, "auto")
            assert _shape(h) == want
            _set(h, "vector", 0, 1)
            assert _shape(h) == (want[0], 1)
            _set(h, "runs")
            assert _shape(h) == (4, 4)
        finally:
            assert _lib.load().gbsp_destroy(h) == 0
