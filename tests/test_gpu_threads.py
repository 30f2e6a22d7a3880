"""Host threads that convert or multiply different matrices at the same time
do not take each other's shared memory: every call succeeds, and its result
is the one the same call gives alone."""
import threading

import numpy as np
import pytest
import torch

from gpu_util import crs, dev, host
from paper_0910_4836_gb300 import synth as S

pytestmark = pytest.mark.gpu
CALLS = 50


@pytest.fixture(scope="module", autouse=True)
def _build():
    import paper_0910_4836_gb300 as g
    g.build()


def _uniform(n, m, length, seed):
    """n rows of `length` entries in m columns."""
    nnz = n * length
    return S.CRS(n, m, (np.arange(n + 1) * length).astype(np.int32),
                 S.randint(seed, 1, np.arange(nnz), 0, m - 1).astype(np.int32), S.vector(nnz, seed))


def _transpose(n, m, length):
    M = crs(_uniform(n, m, length, 11))
    return lambda: [t for T in [M.transpose()] for t in (T.row_ptr, T.col, T.val, T.tmap)]


def _convert(n, length, fmt, **kw):
    M = crs(_uniform(n, n, length, 12))
    return lambda: [t for J in [M.to_jds(fmt, "row_only", **kw)] for t in (J.col, J.val, J.perm, J.blk_ptr)]


def _staged(n, pages):
    A = _uniform(n, n, 9, 13)
    G = crs(A).to_jds("SELL", "row_only", window=128)
    G.stage_x(pages, 1)
    x = dev(S.vector(n, 14))
    return lambda: [G.spmv_original(x)]


# pairs whose launches take more than 48 KB of shared memory, different amounts
PAIRS = {
    "transpose": (lambda: _transpose(2000, 8_000_000, 20), lambda: _transpose(500, 600, 5)),
    "SELL": (lambda: _convert(2000, 25, "SELL", window=256), lambda: _convert(2000, 20, "SELL", window=256)),
    "SOJDS": (lambda: _convert(64, 900, "SOJDS", block=32), lambda: _convert(64, 750, "SOJDS", block=32)),
    "staged x": (lambda: _staged(40_000, 14), lambda: _staged(40_000, 7)),
}


@pytest.mark.parametrize("name", PAIRS)
def test_threads(name):
    large, small = PAIRS[name]
    calls = [large(), small(), small(), small()]
    expect = [[host(t) for t in f()] for f in calls]
    start, faults = threading.Barrier(len(calls)), []

    def work(f, ref):
        try:
            start.wait(60)
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(CALLS):
                    out = f()
                torch.cuda.current_stream().synchronize()
                assert all(np.array_equal(t.cpu().numpy(), r) for t, r in zip(out, ref))
        except BaseException as e:
            faults.append(e)

    threads = [threading.Thread(target=work, args=a) for a in zip(calls, expect)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not faults, faults[0]
