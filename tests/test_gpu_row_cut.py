"""Rows on both sides of the length from which VECTOR takes a row out of its
lane group's loop, which follows the mean row length: against the oracle on
integer data, where any summation order gives the same bits, and the batched
product of the same handles on real data, bit for bit."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import crs, dev, host
from paper_0910_4836_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import paper_0910_4836_gb300 as g
    g.build()


def _matrix(n, base, factor):
    """Rows of `base` entries, every seventh at or around `factor` times the
    mean that they make, or far past it."""
    lens = np.full(n, base, np.int64)
    at = np.arange(3, n, 7)
    cut = factor * base
    for _ in range(20):  # to the fixed point of the mean
        lens[at] = np.resize([cut - 1, cut, cut + 1, 2 * cut, 0, 40 * base], at.size)
        cut = int(factor * lens.sum() / n)
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=row_ptr[1:])
    nnz = int(row_ptr[-1])
    rows = np.repeat(np.arange(n), lens)
    col = (rows * 11 + 17 * (np.arange(nnz) - row_ptr[rows])) % 50_021
    return S.CRS(n, 50_021, row_ptr.astype(np.int32), col.astype(np.int32), S.vector(nnz, 9))


def _check(A, shapes, dtype):
    from paper_0910_4836_gb300 import Batch
    I = S.integer_values(A, 4, 8)
    x, y0 = S.int_vector(A.n_cols, 5, 16), S.int_vector(A.n_rows, 6, 100)
    ref = O.crs_spmv(I, x)
    M, R = crs(I, dtype), crs(A, dtype)
    xd, xr = dev(x, dtype), dev(S.vector(A.n_cols, 8), dtype)
    for shape in shapes:
        for H in (M, R):
            H.set_kernel("vector", lanes=shape[0], rows_per_warp=shape[1])
        assert np.array_equal(host(M.spmv(xd)), ref), shape
        assert np.array_equal(host(M.spmv(xd, out=dev(y0, dtype), accumulate=True)), ref + y0), shape
        y = torch.zeros(A.n_rows, dtype=dtype, device="cuda")
        for chunk in (1000, 4096):
            Batch([(R, xr, y.zero_())], chunk=chunk).run()
            assert torch.equal(y, R.spmv(xr)), (shape, chunk)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("base,factor", [(9, 3), (40, 3), (40, 2), (150, 2), (400, 2)])
def test_cut_by_mean(base, factor, dtype):
    A = _matrix(2003 if base > 100 else 8003, base, factor)
    _check(A, [(l, r) for l in (2, 4, 8, 16, 32) for r in (1, 2, 4)], dtype)


ONE_LANE = [(1, 1), (1, 2), (1, 4)]


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("n", [1, 31, 33, 64, 65, 127, 129, 20_011])
@pytest.mark.parametrize("every", [1, 5, 200])
def test_one_lane_short(n, every, dtype):
    """Short rows with others around the one-lane limits (8 with one set of
    rows a warp, 12 with several) and the warp's (128) in every position; steps
    without any, too."""
    lens = S.randint(3, 1, np.arange(n), 0, 4).astype(np.int64)
    at = np.arange(every // 2, n, every)
    lens[at] = np.resize([8, 9, 12, 13, 0, 128, 129, 300] if every > 1 else [0, 0, 1, 8, 9, 0, 12, 13, 2, 0, 4],
                         at.size)
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=row_ptr[1:])
    nnz = int(row_ptr[-1])
    col = S.randint(7, 1, np.arange(nnz), 0, 50_020)
    _check(S.CRS(n, 50_021, row_ptr.astype(np.int32), col.astype(np.int32), S.vector(nnz, 9)), ONE_LANE, dtype)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("base", [6, 7, 13, 16, 17, 30])
def test_one_lane_asked_for(base, dtype):
    """One lane on longer rows: the limit is twice the mean from 7 to 16."""
    _check(_matrix(4001, base, 2), ONE_LANE, dtype)
