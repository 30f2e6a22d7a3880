"""The fused value gradient for every step count with an instance of its own
and beyond, in both vector layouts, written and accumulated: integer data, where
the fused sums are exact."""
import numpy as np
import pytest
import torch

from gpu_util import adversarial_matrices, crs, dev, host
from paper_0910_4836_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import paper_0910_4836_gb300 as g
    g.build()


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 6, 7, 8, 9, 13])
def test_dval_step_counts(m, dtype):
    for A in adversarial_matrices() + [S.stencil27(9, 4)]:
        if A.nnz == 0:
            continue
        G = np.stack([S.int_vector(A.n_rows, 10 + t, 16) for t in range(m)], 1)
        X = np.stack([S.int_vector(A.n_cols, 40 + t, 16) for t in range(m)], 1)
        d0 = S.int_vector(A.nnz, 3, 100)
        ref = (G[A.row_ids()] * X[A.col]).sum(1)
        M = crs(A, dtype)
        for lay in (lambda a: dev(a, dtype), lambda a: dev(a.T.copy(), dtype).t()):
            assert np.array_equal(host(M.dval_multi(lay(G), lay(X))), ref), A.name
            out = dev(d0, dtype)
            M.dval_multi(lay(G), lay(X), out=out, accumulate=True)
            assert np.array_equal(host(out), d0 + ref), A.name
