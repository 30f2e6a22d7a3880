"""Default lanes of long rows at the limits of the mean row length, in both
types.  Host logic: handles over placeholder addresses."""
import ctypes

import pytest

from paper_0910_4836_gb300 import _lib

P = ctypes.c_void_p(256)  # never dereferenced on the host


def shape(n_rows, nnz, dtype):
    """(lanes, rows) of a new handle."""
    h, o = ctypes.c_void_p(), _lib.KernelOpts()
    assert _lib.load().gbsp_crs_create(n_rows, 64, nnz, P, P, P, dtype, ctypes.byref(h)) == 0
    try:
        assert _lib.load().gbsp_get_kernel(h, ctypes.byref(o)) == 0
        return o.lanes, o.rows_per_warp
    finally:
        assert _lib.load().gbsp_destroy(h) == 0


@pytest.mark.parametrize("mean,f64,f32", [(54, 8, 8), (55, 8, 16), (63, 8, 16), (119, 16, 16), (120, 16, 32),
                                          (191, 16, 32)])
def test_long_rows(mean, f64, f32):
    assert shape(64, 64 * mean, 0) == (f64, 4)
    assert shape(64, 64 * mean, 1) == (f32, 4)


@pytest.mark.parametrize("hundredths,f64,f32", [(0, 1, 1), (1, 4, 4), (149, 4, 4), (150, 2, 4), (224, 2, 4),
                                                (225, 2, 1), (499, 2, 1), (500, 1, 1), (599, 1, 1)])
def test_short_rows(hundredths, f64, f32):
    """Sets of rows a warp with one lane a row, by the mean in hundredths; one
    where there are too few rows for several."""
    for n in (100_000, 99_900):
        nnz = n // 100 * hundredths
        assert shape(n, nnz, 0) == (1, f64 if n == 100_000 else 1)
        assert shape(n, nnz, 1) == (1, f32 if n == 100_000 else 1)
