"""Row-length classes of the CRS kernels (one lane, eight lanes, the whole
warp; rows cut out of a lane group's loop): row lengths on both sides of
every limit, in every position, against the oracle on integer data, where any
summation order gives the same bits; and the batched product of the same
handles on real data, bit for bit."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import crs, dev, host
from paper_0910_4836_gb300 import synth as S

pytestmark = pytest.mark.gpu

LIMITS = (8, 32, 64, 128, 256, 512)  # one lane's, 16 L of 2, 4, 8, 16 and 32 lanes
SHAPES = [(l, r) for l in (1, 2, 4, 8, 16, 32) for r in (1, 2, 4)]


@pytest.fixture(scope="module", autouse=True)
def _build():
    import paper_0910_4836_gb300 as g
    g.build()


def _matrix(n, every):
    """U{0..6} entries a row; every `every`-th row at or around a limit, some
    of several thousand."""
    lens = S.randint(3, 1, np.arange(n), 0, 6).astype(np.int64)
    at = np.arange(0, n, every)
    pick = np.array([l + d for l in LIMITS for d in (-1, 0, 1)] + [1531, 2999])
    lens[at] = pick[np.arange(at.size) % pick.size]
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=row_ptr[1:])
    nnz = int(row_ptr[-1])
    rows = np.repeat(np.arange(n), lens)
    col = (rows * 11 + 17 * (np.arange(nnz) - row_ptr[rows])) % 50_021
    return S.CRS(n, 50_021, row_ptr.astype(np.int32), col.astype(np.int32), S.vector(nnz, 9))


@pytest.mark.parametrize("n,every", [(1, 1), (33, 2), (2001, 1), (20_011, 7), (20_011, 97)])
def test_row_classes(n, every):
    A = S.integer_values(_matrix(n, every), 4, 8)
    x = S.int_vector(A.n_cols, 5, 16)
    y0 = S.int_vector(n, 6, 100)
    ref = O.crs_spmv(A, x)
    for dtype in (torch.float64, torch.float32):  # sums below 2^24: exact in both
        M = crs(A, dtype)
        xd, yd = dev(x, dtype), dev(y0, dtype)
        X2 = torch.stack([xd, xd.flip(0)], 1)
        for l, r in SHAPES:
            M.set_kernel("vector", lanes=l, rows_per_warp=r)
            assert np.array_equal(host(M.spmv(xd)), ref), (l, r)
            assert np.array_equal(host(M.spmv(xd, out=yd.clone(), accumulate=True)), ref + y0), (l, r)
            # a strided column in and out
            Y2 = torch.zeros((n, 2), dtype=dtype, device="cuda")
            M.spmm(X2[:, :1], out=Y2[:, 1:])
            assert np.array_equal(host(Y2[:, 1]), ref) and not host(Y2[:, 0]).any(), (l, r)
        for l, r in ((2, 4), (4, 4), (8, 8)):
            M.set_kernel("runs", lanes=l, rows_per_warp=r)
            assert np.array_equal(host(M.spmv(xd)), ref), ("runs", l, r)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_row_classes_batched(dtype):
    from paper_0910_4836_gb300 import Batch
    A = _matrix(20_011, 7)
    x = dev(S.vector(A.n_cols, 8), dtype)
    items, refs = [], []
    for l, r in SHAPES:
        M = crs(A, dtype)
        M.set_kernel("vector", lanes=l, rows_per_warp=r)
        items.append((M, x, torch.zeros(A.n_rows, dtype=dtype, device="cuda")))
        refs.append(M.spmv(x))
    for chunk in (1000, 4096):
        Batch(items, chunk=chunk).run()
        for (_, _, y), ref, shape in zip(items, refs, SHAPES):
            assert torch.equal(y, ref), (shape, chunk)
            y.zero_()
