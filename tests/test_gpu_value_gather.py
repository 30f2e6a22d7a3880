"""Re-gathered values of JDS and SELL storage on rows of one entry and fewer,
where a slot at a time is gathered, and on either side of 1.5 entries a row:
the same bytes as a conversion of the matrix with those values."""
import numpy as np
import pytest
import torch

from gpu_util import crs, dev, host
from paper_0910_4836_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import paper_0910_4836_gb300 as g
    g.build()


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("fmt", ["NUJDS", "JDS", "SELL"])
@pytest.mark.parametrize("lens", [[1], [0, 1], [1, 2], [2, 1, 1], [0, 9, 1, 1, 0, 0], [5]])
def test_refreshed_values(lens, fmt, dtype):
    n = 3001
    lens = np.resize(lens, n).astype(np.int64)
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=row_ptr[1:])
    nnz = int(row_ptr[-1])
    A = S.CRS(n, n, row_ptr.astype(np.int32), S.randint(7, 1, np.arange(nnz), 0, n - 1).astype(np.int32),
              S.vector(nnz, 9))
    J = crs(A, dtype).to_jds(fmt, "row_only", window=128, value_map=True)
    B = S.CRS(n, n, A.row_ptr, A.col, S.vector(nnz, 10))
    J.refresh_values(dev(B.val, dtype))
    assert np.array_equal(host(J.val), host(crs(B, dtype).to_jds(fmt, "row_only", window=128).val))
