"""SpMM at row counts where the rows a warp takes change (from its groups' one
round to sixteen): against the oracle on integer data, and bit for bit against
the batched product, whose warps take other rows."""
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


@pytest.mark.parametrize("n", [1, 19_455, 40_001, 70_003, 120_001, 320_011])
def test_rows_a_warp(n):
    from paper_0910_4836_gb300 import Batch
    lens = S.randint(3, 1, np.arange(n), 0, 9).astype(np.int64)
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=row_ptr[1:])
    nnz = int(row_ptr[-1])
    A = S.CRS(n, 5003, row_ptr.astype(np.int32), S.randint(7, 1, np.arange(nnz), 0, 5002).astype(np.int32),
              S.vector(nnz, 9))
    I = S.integer_values(A, 4, 8)
    M, R = crs(I), crs(A)
    x = [S.int_vector(A.n_cols, 30 + j, 16) for j in range(20)]
    ref = [O.crs_spmv(I, v) for v in x]
    for k, tile in ((3, 16), (5, 16), (16, 16), (20, 16), (20, 32)):
        for H in (M, R):
            H.set_kernel("vector", rhs_tile=tile)
        Y = host(M.spmm(dev(np.stack(x[:k], 1))))
        assert all(np.array_equal(Y[:, j], ref[j]) for j in range(k)), (k, tile)
        X = dev(S.vector(A.n_cols * k, 8).reshape(-1, k))
        B = torch.zeros((n, k), dtype=torch.float64, device="cuda")
        Batch([(R, X, B)]).run()
        assert torch.equal(B, R.spmm(X)), (k, tile)
