"""CRS products with k right-hand sides at every lane-group width, pass count
and edge of a warp's row set: integer data, where any summation order gives
the oracle's bits, and the batched product on real data bit for bit."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import crs, dev, host
from paper_0910_4836_gb300 import synth as S

pytestmark = pytest.mark.gpu

KS = (2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 15, 16, 17, 20, 31, 32, 33, 40)


@pytest.fixture(scope="module", autouse=True)
def _build():
    import paper_0910_4836_gb300 as g
    g.build()


def _matrix(n):
    """Rows of 0 to 9 entries, every eleventh of up to 70."""
    lens = S.randint(3, 1, np.arange(n), 0, 9).astype(np.int64)
    lens[::11] = S.randint(3, 2, np.arange(lens[::11].size), 0, 70)
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=row_ptr[1:])
    nnz = int(row_ptr[-1])
    rows = np.repeat(np.arange(n), lens)
    col = (rows * 3 + 5 * (np.arange(nnz) - row_ptr[rows])) % 997
    return S.CRS(n, 997, row_ptr.astype(np.int32), col.astype(np.int32), S.vector(nnz, 9))


@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 33, 1000, 5003])
def test_spmm_widths(n):
    A = S.integer_values(_matrix(n), 4, 8)
    X = np.stack([S.int_vector(A.n_cols, 5 + c, 16) for c in range(max(KS))], 1)
    Y0 = np.stack([S.int_vector(n, 70 + c, 100) for c in range(max(KS))], 1)
    ref = O.crs_spmm(A, X)
    for dtype in (torch.float64, torch.float32):
        M = crs(A, dtype)
        Xd, Yd = dev(X, dtype), dev(Y0, dtype)
        for k in KS:
            for tile in (0, 4, 32) if n in (33, 1000) else (0,):
                M.set_kernel("vector", rhs_tile=tile)
                # leading dimensions wider than k
                assert np.array_equal(host(M.spmm(Xd[:, :k])), ref[:, :k]), (dtype, k, tile)
                Y = Yd.clone()
                M.spmm(Xd[:, :k].contiguous(), out=Y[:, :k], accumulate=True)
                assert np.array_equal(host(Y[:, :k]), ref[:, :k] + Y0[:, :k]), (dtype, k, tile)
                assert np.array_equal(host(Y[:, k:]), Y0[:, k:]), (dtype, k, tile)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("jds", [False, True])
def test_spmm_widths_batched(dtype, jds):
    """Batches of CRS items alone, and beside SELL items with one and with
    several right-hand sides (the other kernel instances)."""
    from paper_0910_4836_gb300 import Batch
    items, refs = [], []
    for i, k in enumerate((1,) + KS if jds else KS):
        A = _matrix(400 + 7 * i)
        H = crs(A, dtype)
        if jds and i % 3 == 0:
            H = H.to_jds("SELL", "row_only", window=128)
        X = dev(np.stack([S.vector(A.n_cols, 20 + c) for c in range(k)], 1), dtype)
        items.append((H, X, torch.zeros((A.n_rows, k), dtype=dtype, device="cuda")))
        refs.append(H.spmm(X))
    for n in (len(items), 4):  # all, and the narrow ones (k <= 4)
        Batch(items[:n], chunk=1000).run()
        for (_, _, Y), ref in zip(items[:n], refs):
            assert torch.equal(Y, ref)
            Y.zero_()
