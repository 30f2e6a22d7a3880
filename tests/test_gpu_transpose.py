"""The column-split transpose at the edges of its buckets, rounds and sizes:
bit-exact against a stable sort of the entries by column."""
import numpy as np
import pytest
import torch

from gpu_util import crs, host
from paper_0910_4836_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import paper_0910_4836_gb300 as g
    g.build()


def _matrix(n, m, lens, cols):
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=row_ptr[1:])
    nnz = int(row_ptr[-1])
    return S.CRS(n, m, row_ptr.astype(np.int32), cols(nnz).astype(np.int32), S.vector(nnz, 5))


def _uniform(m):
    return lambda k: S.randint(7, 1, np.arange(k), 0, m - 1)


CASES = {
    "one entry": lambda: _matrix(1, 1, [1], _uniform(1)),
    "fewer columns than lanes": lambda: _matrix(50_000, 3, S.randint(1, 1, np.arange(50_000), 0, 5), _uniform(3)),
    "empty rows and columns": lambda: _matrix(7001, 9001, S.randint(2, 1, np.arange(7001), 0, 2), _uniform(9001)),
    # one column's records span several rounds of a bucket
    "one dense column": lambda: _matrix(40_001, 300_000, np.ones(40_001, np.int64), lambda k: np.full(k, 123_457)),
    # columns around the length from which a warp collects them
    "columns of 47 to 50": lambda: _matrix(50, 2000, np.full(50, 1900), lambda k: np.concatenate(
        [(np.arange(1900) + (r if r > 46 else 0)) % 2000 for r in range(50)])),
    "one dense row": lambda: _matrix(3, 70_000, [0, 200_003, 1], _uniform(70_000)),
    # the last column count of the split and the first of the radix sort
    "2^24 columns": lambda: _matrix(1000, 1 << 24, np.full(1000, 11), _uniform(1 << 24)),
    "2^24 + 1 columns": lambda: _matrix(1000, (1 << 24) + 1, np.full(1000, 11), _uniform((1 << 24) + 1)),
}


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("name", CASES)
def test_transpose_edges(name, dtype):
    A = CASES[name]()
    T = crs(A, dtype).transpose()
    order = np.argsort(A.col, kind="stable")
    row_ptr = np.zeros(A.n_cols + 1, np.int64)
    np.cumsum(np.bincount(A.col, minlength=A.n_cols), out=row_ptr[1:])
    assert np.array_equal(host(T.row_ptr), row_ptr)
    assert np.array_equal(host(T.tmap), order)
    assert np.array_equal(host(T.col), A.row_ids()[order])
    assert np.array_equal(host(T.val), A.val.astype(host(T.val).dtype)[order])
