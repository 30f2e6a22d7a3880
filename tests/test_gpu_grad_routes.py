"""Gradients through a Pattern whose values move, are not contiguous, or need
only one of the two gradients: against the products written out in FP64."""
import numpy as np
import pytest
import torch

from gpu_util import dev, host
from paper_0910_4836_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import paper_0910_4836_gb300 as g
    g.build()


def _pattern(A, **kw):
    from paper_0910_4836_gb300.autograd import Pattern
    return Pattern.from_host(A, **kw)


def _dx(A, val, g):
    """A^T g and the sum of |a||g| that its rounding is measured by."""
    out, s = np.zeros(A.n_cols), np.zeros(A.n_cols)
    p = val * g[A.row_ids()]
    np.add.at(out, A.col, p)
    np.add.at(s, A.col, np.abs(p))
    return out, s


@pytest.mark.parametrize("kind", ["crs", "jds", "sell"])
def test_values_in_reused_memory(kind):
    """v1 forward and backward, v2 forward, then v3 in v1's freed memory with
    v1's version: y and dx are v3's."""
    from paper_0910_4836_gb300.autograd import spmv
    A = S.small_random(3000, 3000, 81, density=0.004)
    P = _pattern(A, adjoint=kind, forward=kind)
    x, g = S.vector(A.n_cols, 82), S.vector(A.n_rows, 83)
    xd, gd = dev(x).requires_grad_(), dev(g)
    values = [S.vector(A.nnz, s) for s in (84, 85, 86)]
    staged = [dev(v) for v in values]
    v1 = staged[0].clone()
    at, version = v1.data_ptr(), v1._version
    torch.autograd.grad(spmv(P, v1, xd), xd, gd)
    v2 = staged[1].clone()
    spmv(P, v2, xd.detach())
    torch.cuda.synchronize()
    del v1
    v3 = staged[2].clone()
    if (v3.data_ptr(), v3._version) != (at, version):
        pytest.skip("the allocator gave other memory")
    y = spmv(P, v3, xd)
    dx, = torch.autograd.grad(y, xd, gd)
    ref, s = _dx(A, values[2], g)
    assert np.all(np.abs(host(dx) - ref) <= 1e-14 * s + 1e-300)
    T = S.CRS(A.n_rows, A.n_cols, A.row_ptr, A.col, values[2])
    yref = np.zeros(A.n_rows)
    np.add.at(yref, A.row_ids(), T.val * x[A.col])
    ys = np.zeros(A.n_rows)
    np.add.at(ys, A.row_ids(), np.abs(T.val * x[A.col]))
    assert np.all(np.abs(host(y) - yref) <= 1e-14 * ys + 1e-300)


@pytest.mark.parametrize("kind", ["crs", "jds", "sell"])
def test_values_not_contiguous(kind):
    """A strided view of changing memory is read anew by every call."""
    from paper_0910_4836_gb300.autograd import spmv
    A = S.small_random(2000, 2000, 87, density=0.004)
    P = _pattern(A, adjoint=kind, forward=kind)
    xd, g = dev(S.vector(A.n_cols, 88)).requires_grad_(), S.vector(A.n_rows, 89)
    for seed in (90, 91):
        pair = np.stack([S.vector(A.nnz, seed), np.full(A.nnz, np.nan)], 1)
        dx, = torch.autograd.grad(spmv(P, dev(pair)[:, 0], xd), xd, dev(g))
        ref, s = _dx(A, pair[:, 0], g)
        assert np.all(np.abs(host(dx) - ref) <= 1e-14 * s + 1e-300)


def test_handle_pointed_elsewhere_between_calls():
    """The caller moves the pattern's own CRS handle and re-gathers A^T from
    there; the next backward pass uses its own values again."""
    from paper_0910_4836_gb300.autograd import spmv
    A = S.small_random(2000, 2000, 92, density=0.004)
    P = _pattern(A)
    x, g = dev(S.vector(A.n_cols, 93)).requires_grad_(), S.vector(A.n_rows, 94)
    v = S.vector(A.nnz, 95)
    val, other = dev(v), dev(S.vector(A.nnz, 96))
    torch.autograd.grad(spmv(P, val, x), x, dev(g))
    P.A.set_values(other)
    P.A.refresh_transpose_values()
    dx, = torch.autograd.grad(spmv(P, val, x), x, dev(g))
    ref, s = _dx(A, v, g)
    assert np.all(np.abs(host(dx) - ref) <= 1e-14 * s + 1e-300)


M, N = 20, 50_000


def _power_pattern():
    A = S.hh_like(N, 97)
    val = dev(A.val / 64)
    return A, _pattern(A), val


@pytest.mark.parametrize("checkpoint", [1, 2, 5, 7, 12, 20, 30])
def test_power_memory(checkpoint):
    """Between forward and backward a call holds y and at most twice its
    checkpoints, x among them, but x alone with checkpoint >= m; two calls in
    one graph hold twice that, and no_grad holds y alone."""
    from paper_0910_4836_gb300.autograd import power_apply
    _, P, val = _power_pattern()
    x = dev(S.vector(N, 98)).requires_grad_()
    val.requires_grad_()
    power_apply(P, val, x, 2, 1)
    vector = N * 8 + 2048  # the allocator's rounding
    held = 0 if checkpoint >= M else 2 * -(-M // checkpoint) - 1
    for calls, grad in ((1, True), (2, True), (1, False)):
        torch.cuda.synchronize()
        before = torch.cuda.memory_allocated()
        with torch.set_grad_enabled(grad):
            ys = [power_apply(P, val, x, M, checkpoint) for _ in range(calls)]
        assert torch.cuda.memory_allocated() - before <= calls * (1 + (held if grad else 0)) * vector
        del ys


@pytest.mark.parametrize("checkpoint", [2, 5, 20])
def test_power_peak(checkpoint):
    """The backward pass takes three segments, the value gradient and dx
    beyond what the checkpoints hold."""
    from paper_0910_4836_gb300.autograd import power_apply
    A, P, val = _power_pattern()
    x, g = dev(S.vector(N, 98)).requires_grad_(), dev(S.vector(N, 99))
    val.requires_grad_()
    torch.autograd.grad(power_apply(P, val, x, M, checkpoint), (val, x), g)
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    torch.cuda.reset_peak_memory_stats()
    torch.autograd.grad(power_apply(P, val, x, M, checkpoint), (val, x), g)
    peak = torch.cuda.max_memory_allocated() - before - A.nnz * 8
    assert peak <= (3 * checkpoint + -(-M // checkpoint) + 1) * (N * 8 + 2048)


@pytest.mark.parametrize("checkpoint", [1, 3, 5, 20])
@pytest.mark.parametrize("needs", ["values", "x"])
def test_power_one_gradient(needs, checkpoint):
    """A gradient asked for alone has the bits it has beside the other."""
    from paper_0910_4836_gb300.autograd import power_apply
    _, P, val = _power_pattern()
    g, xv = dev(S.vector(N, 99)), dev(S.vector(N, 98))
    both = [val.clone().requires_grad_(), xv.clone().requires_grad_()]
    ref = torch.autograd.grad(power_apply(P, *both, M, checkpoint), both, g)
    at = 0 if needs == "values" else 1
    one = [val, xv]
    one[at] = one[at].clone().requires_grad_()
    got, = torch.autograd.grad(power_apply(P, *one, M, checkpoint), one[at], g)
    assert torch.equal(got, ref[at])
