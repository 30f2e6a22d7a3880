"""The split JDS walk with few and with many chunks (more than a CTA counts at
once), every unroll depth, both bases, strided vectors: integer data, where any
summation order gives the oracle's bits."""
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


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("perm", ["symmetric", "row_only"])
def test_split_walk_chunks(perm, dtype):
    n = 3001
    lens = S.randint(5, 1, np.arange(n), 0, 12).astype(np.int64)
    lens[::37] = S.randint(5, 2, np.arange(lens[::37].size), 13, 90)
    lens[[5, 700, 2999]] = (1500, 1499, 600)
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=row_ptr[1:])
    nnz = int(row_ptr[-1])
    A = S.CRS(n, n, row_ptr.astype(np.int32), S.randint(3, 1, np.arange(nnz), 0, n - 1).astype(np.int32),
              (np.arange(nnz) % 9 - 4).astype(np.float64))
    x = S.int_vector(n, 3, 8)
    y0 = S.int_vector(n, 4, 50)
    ref = O.crs_spmv(A, x)
    xd, yd = dev(x, dtype), dev(y0, dtype)
    X2 = torch.stack([xd.flip(0), xd], 1)
    for unroll in (1, 2, 4, 8, 16):
        J = crs(A, dtype).to_jds("NUJDS", perm, unroll=unroll)
        for depth, chunk in ((16, 64), (2, 4), (12, 1), (89, 500), (1499, 7)):
            J.split(depth, chunk)
            assert np.array_equal(host(J.spmv_original(xd)), ref), (unroll, depth, chunk)
            assert np.array_equal(host(J.spmv_original(xd, out=yd.clone(), accumulate=True)), ref + y0)
            xp = J.permute(xd) if perm == "symmetric" else xd
            assert np.array_equal(host(J.permute(J.spmv(xp), back=True)), ref), (unroll, depth, chunk)
            Y2 = torch.zeros((n, 2), dtype=dtype, device="cuda")
            J.spmm(X2[:, 1:], out=Y2[:, :1], basis=1)
            assert np.array_equal(host(Y2[:, 0]), ref), (unroll, depth, chunk)


@pytest.mark.parametrize("unroll", [1, 8, 16])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_split_apart(unroll, dtype):
    """Deep items enough to fill the GPU, on rows most of which go deep: the
    deep items are launched before the walk.  Integer data, any order exact."""
    n = 400_000 if unroll == 1 else 60_000
    lens = S.randint(3, 1, np.arange(n), 0, 50).astype(np.int64)
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=row_ptr[1:])
    nnz = int(row_ptr[-1])
    A = S.integer_values(S.CRS(n, n, row_ptr.astype(np.int32), S.randint(7, 1, np.arange(nnz), 0, n - 1).astype(
        np.int32), S.vector(nnz, 9)), 4, 8)
    x, y0 = S.int_vector(n, 5, 16), S.int_vector(n, 6, 100)
    ref = O.crs_spmv(A, x)
    J = crs(A, dtype).to_jds("NUJDS", "symmetric", unroll=unroll)
    for depth, chunk in ((1, 1), (9, 1), (30, 1), (49, 8)):  # (30, 1): few entries deep
        J.split(depth, chunk)
        for limit in (0, 3):
            J.set_grid_limit(limit)
            assert np.array_equal(host(J.spmv_original(dev(x, dtype))), ref), (depth, chunk, limit)
            y = J.spmv(J.permute(dev(x, dtype)), out=J.permute(dev(y0, dtype)), accumulate=True)
            assert np.array_equal(host(J.permute(y, back=True)), ref + y0), (depth, chunk, limit)
