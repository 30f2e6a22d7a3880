"""Transposes of long rows, whose entries find their row tile by tile, and of
columns of every length class of a bucket's round: bit-exact against a stable
sort of the entries by column."""
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


def _check(n, m, lens, cols, dtype):
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=row_ptr[1:])
    nnz = int(row_ptr[-1])
    A = S.CRS(n, m, row_ptr.astype(np.int32), cols(nnz).astype(np.int32), S.vector(nnz, 5))
    T = crs(A, dtype).transpose()
    order = np.argsort(A.col, kind="stable")
    t_row_ptr = np.zeros(m + 1, np.int64)
    np.cumsum(np.bincount(A.col, minlength=m), out=t_row_ptr[1:])
    assert np.array_equal(host(T.row_ptr), t_row_ptr)
    assert np.array_equal(host(T.tmap), order)
    assert np.array_equal(host(T.col), A.row_ids()[order])
    assert np.array_equal(host(T.val), A.val.astype(host(T.val).dtype)[order])


ROWS = {
    "one row": [70_001],
    "tile edges": [2047, 1, 2048, 2049, 0, 0, 4096, 1],
    "empty rows at tile edges": [0, 0, 2048, 0, 0, 0, 4095, 0, 1, 0, 2048, 0, 0],
    "long and empty": np.where(np.arange(3000) % 50 == 7, 7001, 0),
    "many short, a few very long": np.where(np.arange(40_000) % 20_000 == 11, 3_000_000, 1),
    "mean 128": np.full(700, 128),
    "mean below 128": np.full(700, 127),
}


@pytest.mark.parametrize("columns", [20_000, (1 << 24) + 1])  # column split, radix sort
@pytest.mark.parametrize("name", ROWS)
def test_long_rows(name, columns):
    lens = np.asarray(ROWS[name], np.int64)
    _check(lens.size, columns, lens, lambda k: S.randint(7, 1, np.arange(k), 0, columns - 1), torch.float64)


@pytest.mark.parametrize("nnz", [(1 << 20) - 1, 1 << 20, 2_500_001])
@pytest.mark.parametrize("columns", [1, 2])
def test_few_columns(columns, nnz):
    """2^20 entries a column and more go to the radix sort."""
    lens = np.resize([7, 0, 3, 11], nnz // 5)
    lens = lens[np.cumsum(lens) <= nnz]
    lens = np.append(lens, nnz - lens.sum())
    _check(lens.size, columns, lens, lambda k: S.randint(7, 1, np.arange(k), 0, columns - 1), torch.float64)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("longest", [47, 49, 64, 97, 127, 128, 129, 160, 300])
def test_column_lengths(longest, dtype):
    """Columns of `longest` - 2 to `longest` entries (one thread to 48, a warp's
    ranks to 128, a warp's pass over the round from 129), shuffled over rows."""
    m = 400
    count = longest - np.arange(m) % 3
    col = np.repeat(np.arange(m), count)
    rng = np.random.default_rng(3)
    rng.shuffle(col)
    lens = np.bincount(rng.integers(0, 5000, col.size), minlength=5000)
    _check(5000, m, lens, lambda k: col, dtype)
