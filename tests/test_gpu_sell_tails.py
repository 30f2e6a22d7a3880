"""The last step of the SELL walk: blocks whose longest row leaves any number
of slots, on both sides of the size rule that picks the exact last step.
Integer data, where any summation order gives the oracle's bits."""
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


def _matrix(lens, n_cols):
    row_ptr = np.zeros(lens.size + 1, np.int64)
    np.cumsum(lens, out=row_ptr[1:])
    nnz = int(row_ptr[-1])
    rows = np.repeat(np.arange(lens.size), lens)
    col = (rows + 7 * (np.arange(nnz) - row_ptr[rows])) % n_cols
    val = (np.arange(nnz) % 17 - 8).astype(np.float64)
    return S.CRS(lens.size, n_cols, row_ptr.astype(np.int32), col.astype(np.int32), val)


@pytest.mark.parametrize("unroll", [1, 2, 4])
def test_sell_last_step(unroll):
    from paper_0910_4836_gb300 import Batch
    # 32-row blocks whose longest row has 0, 1, ... 13 entries, the last partial
    lens = np.concatenate([np.maximum(w - np.arange(32) % 5, 0) for w in range(14)])[:-3]
    A = _matrix(lens, 211)
    x = S.int_vector(211, 3, 16)
    ref = O.crs_spmv(A, x)
    for dtype in (torch.float64, torch.float32):
        G = crs(A, dtype).to_jds("SELL", "row_only", window=32, unroll=unroll)
        xd = dev(x, dtype)
        assert np.array_equal(host(G.spmv_original(xd)), ref)
        y = torch.ones(lens.size, dtype=dtype, device="cuda")
        G.spmv(xd, out=y, accumulate=True)
        assert np.array_equal(host(G.permute(y, back=True)), ref + 1)
        X = torch.stack([xd, -xd, 2 * xd], 1)
        assert np.array_equal(host(G.spmm(X, basis=1)), np.stack([ref, -ref, 2 * ref], 1))
        y.zero_()
        Batch([(G, xd, y)], chunk=64).run()
        assert np.array_equal(host(G.permute(y, back=True)), ref)


@pytest.mark.parametrize("n", [(1 << 22) - 5, (1 << 22) + 37])  # y of just under and just over 32 MB
def test_sell_last_step_rule(n):
    A = _matrix(S.randint(5, 1, np.arange(n), 0, 6).astype(np.int64), n)
    x = S.int_vector(n, 3, 16)
    G = crs(A).to_jds("SELL", "row_only", window=64, unroll=4)
    assert np.array_equal(host(G.spmv_original(dev(x))), O.crs_spmv(A, x))
