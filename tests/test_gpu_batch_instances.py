"""Every kernel instance of the batch: batches of one type and of both, with
and without CRS items of one and of several right-hand sides, and JDS-family
items of up to four and of more: each result has the bits of its product
alone."""
import pytest
import torch

from gpu_util import crs, dev
from paper_0910_4836_gb300 import synth as S

pytestmark = pytest.mark.gpu
F64, F32 = torch.float64, torch.float32


@pytest.fixture(scope="module", autouse=True)
def _build():
    import paper_0910_4836_gb300 as g
    g.build()


@pytest.mark.parametrize("compensated", [True, False])
@pytest.mark.parametrize("kinds", [("crs1",), ("crs1", "crs5"), ("crs4", "sell1"), ("sell4",), ("jds4", "sell3"),
                                   ("crs1", "jds4"), ("crs2", "sell4"), ("jds7", "crs1"), ("sell16", "crs16", "crs1")])
@pytest.mark.parametrize("types", [(F64,), (F32,), (F64, F32)])
def test_instances(kinds, types, compensated):
    from paper_0910_4836_gb300 import Batch
    items = []
    for i in range(6):
        kind, dtype = kinds[i % len(kinds)], types[i % len(types)]
        fmt, k = kind.rstrip("0123456789"), int(kind.lstrip("abcdefghijklmnopqrstuvwxyz"))
        M = crs(S.zipf_rows(3000 + 517 * i, 20 + i, lmax=400), dtype)
        if dtype == F32:
            M.set_kernel("vector", compensated=compensated)
        H = M if fmt == "crs" else M.to_jds(fmt.upper(), "row_only", window=128)
        n = M.n_rows
        x = dev(S.vector(n * k, 40 + i), dtype)
        items.append((H, x if k == 1 else x.reshape(n, k), torch.zeros((n,) if k == 1 else (n, k), dtype=dtype,
                                                                       device="cuda")))
    Batch(items).run()
    for i, (H, x, y) in enumerate(items):
        assert torch.equal(y, H.spmm(x)), (i, kinds[i % len(kinds)])
