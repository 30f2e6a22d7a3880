"""CRS -> SELL / JDS conversion at the edges of its sorts and copies, bit-exact
against the oracle's builders: windows on both sides of the one-launch sort
and of the staged copy, rows longer than a key, a block's near slots or a
thread's share, partial windows, arrays off a 16-byte boundary."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import crs, host
from paper_0910_4836_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import paper_0910_4836_gb300 as g
    g.build()


def _matrix(lens):
    lens = np.asarray(lens, np.int64)
    n = lens.size
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=row_ptr[1:])
    nnz = int(row_ptr[-1])
    return S.CRS(n, n, row_ptr.astype(np.int32), S.randint(3, 1, np.arange(nnz), 0, n - 1).astype(np.int32),
                 S.vector(nnz, 4))


def _lengths(n, long):
    lens = S.randint(5, 1, np.arange(n), 0, 12).astype(np.int64)
    at = S.randint(5, 2, np.arange(len(long)), 0, n - 1)
    lens[at] = long
    return lens


ROWS = {
    "one row": [3],
    "all equal": [5] * 1000,
    "around the near slots": _lengths(1500, [30, 31, 32, 33, 63, 64, 65, 66, 64, 65, 200, 201, 199]),
    "heavy tail": _lengths(5003, [4000, 3999, 700, 701, 64, 2500]),
    "a row past a sort key": _lengths(500, [(1 << 20) + 3, 1 << 20, (1 << 20) - 1]),
    "windows of very different sizes": np.repeat([0, 1, 40, 2, 0, 25], 700),
}


@pytest.mark.parametrize("perm", ["symmetric", "row_only"])
@pytest.mark.parametrize("name", ROWS)
def test_sell_build_edges(name, perm):
    A = _matrix(ROWS[name])
    M = crs(A)
    for window in (32, 96, 128, 256, 288, 1024, 1056):
        Os = O.sell_build(A, window, symmetric=perm == "symmetric")
        G = M.to_jds("SELL", perm, window=window, value_map=True)
        for k in ("perm", "iperm", "rlen", "blk_ptr", "col", "val"):
            assert np.array_equal(host(getattr(G, k)), getattr(Os, k)), (window, k)
        assert np.array_equal(A.val[host(G.vmap)], Os.val), window


@pytest.mark.parametrize("perm", ["symmetric", "row_only"])
@pytest.mark.parametrize("name", [k for k in ROWS if k != "a row past a sort key"])
def test_jds_build_edges(name, perm):
    A = _matrix(ROWS[name])
    Oj = O.jds_build(A, perm == "symmetric")
    J = crs(A).to_jds("JDS", perm, value_map=True)
    for k in ("perm", "iperm", "jd_ptr", "col", "val"):
        assert np.array_equal(host(getattr(J, k)), getattr(Oj, k)), k
    assert np.array_equal(A.val[host(J.vmap)], Oj.val)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_sell_build_unaligned_arrays(dtype):
    from paper_0910_4836_gb300 import CRSMatrix
    A = _matrix(ROWS["windows of very different sizes"])
    Os = O.sell_build(A, 128)
    val = torch.as_tensor(A.val).to(dtype)
    for lead in (0, 1, 2, 3):
        col_d = torch.cat([torch.zeros(lead, dtype=torch.int32), torch.as_tensor(A.col)]).cuda()[lead:]
        val_d = torch.cat([torch.zeros(lead, dtype=dtype), val]).cuda()[lead:]
        G = CRSMatrix(torch.as_tensor(A.row_ptr).cuda(), col_d, val_d, A.n_cols).to_jds("SELL", "symmetric", window=128)
        assert np.array_equal(host(G.col), Os.col), lead
        assert np.array_equal(host(G.val), Os.val.astype(host(G.val).dtype)), lead


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("name", ROWS)
def test_value_refresh_edges(name, dtype):
    A = _matrix(ROWS[name])
    M = crs(A, dtype)
    T = M.transpose()
    handles = [T.to_jds(f, "row_only", window=128, value_map=True) for f in ("SELL", "NUJDS")]
    new = torch.as_tensor(S.vector(A.nnz, 8)).to(dtype).cuda()
    M.set_values(new)
    M.refresh_transpose_values()
    assert torch.equal(T.val, new[T.tmap.long()])
    for H in handles:
        H.refresh_values(T.val)
        assert torch.equal(H.val, T.val[H.vmap.long()]), H.fmt
