"""The autotuner's candidates cover what a handle takes by itself: one lane a
row on short rows, and one row a thread on a split walk, whose tuning is its
own."""
import pytest
import torch

from gpu_util import crs, dev, host
from paper_0910_4836_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import paper_0910_4836_gb300 as g
    g.build()


def test_one_lane_is_tried():
    """Two lanes a row take a third longer than one on this grid."""
    M = crs(S.laplace2d(1500, 1500))
    best, ms = M.autotune()
    assert best["lanes"] == 1 and ms > 0


def test_split_walk():
    A = S.zipf_rows(60_000, 9, lmax=3000)
    M = crs(A)
    J = M.to_jds("NUJDS", "symmetric", unroll=2)
    x = J.permute(dev(S.vector(A.n_cols, 5)))
    J.split(16, 64)
    best, ms = J.autotune()
    assert best["rows_per_warp"] == 1
    y = J.spmv(x)
    J.split(0)
    _, unsplit = J.autotune()
    assert unsplit > 1.5 * ms  # 3000 diagonals one after another, not the split's cached time
    assert torch.allclose(y, J.spmv(x), rtol=1e-12, atol=1e-12)
