"""The sparse products, gradients and conversions that this library is timed on.

Each case is one call (or one training step) as a program makes it through
the Python classes: a matrix of one of the repository's workload recipes,
made on the GPU, in the storage scheme such a program keeps.  A case fixes
the sizes of its matrices, entry counts among them; the seed gives their
entries (the recipe's pattern under a shift of the index range, the values)
and the vectors.

  op      spmv       y = A x through a kept handle
          spmm       Y = A X, k right-hand sides
          grad       y = A x, then the gradients for A's values and for x
          power      a training step on y = A^m x: forward, checkpointed
                     backward, update of the values
          batch      one persistent launch over many matrices
          convert    CRS -> SELL-32-sigma / NUJDS
          transpose  CRS of A^T with its entry map
  matrix  hh         banded-plus-scattered, ~13 entries a row (Sect. 4.2)
          zipf       heavy-tailed row lengths, uniform columns
          stencil27  27-point stencil on an m^3 grid
          laplace    5-point Laplacian on an m x m grid
          random     U{5..30} entries a row, uniform columns
"""
import math

import torch

from paper_0910_4836_gb300.autograd import Pattern, power_apply, spmv
from paper_0910_4836_gb300.batch import Batch
from paper_0910_4836_gb300.sparse import CRSMatrix

DEV = "cuda"
DTYPES = {"f64": torch.float64, "f32": torch.float32}
HH_OFFSETS = (1, 256, 512, 768, 1024, 65536, 131072, 196608, 262144)
SPLIT_DEPTH, SPLIT_CHUNK = 16, 64  # the benchmark's deep split for the Zipf rows
LEARNING_RATE = 1e-6


def listed():
    return [
        # The smallest call: one product of an iterative solver on a small
        # grid, bound by the launch and the call itself.
        {"name": "laplace64_crs", "op": "spmv", "matrix": "laplace", "n": 64, "format": "crs", "dtype": "f64"},
        # The benchmark's step: an eigensolver's product in the permuted
        # basis, matrix and vectors far larger than L2.
        {"name": "hh6M_sell_step", "op": "spmv", "matrix": "hh", "n": 6000000, "format": "sell_sym", "dtype": "f64"},
        # The same kind of matrix at the paper's dimension, in plain CRS
        # without any set-up or tuning.
        {"name": "hh1M2_crs", "op": "spmv", "matrix": "hh", "n": 1201200, "format": "crs", "dtype": "f64"},
        # Irregular rows (a graph) in plain CRS.
        {"name": "zipf4M_crs", "op": "spmv", "matrix": "zipf", "n": 4000000, "format": "crs", "dtype": "f64"},
        # The same rows in the tuned storage for heavy tails.
        {"name": "zipf4M_nujds_split", "op": "spmv", "matrix": "zipf", "n": 4000000, "format": "nujds_split",
         "dtype": "f64"},
        # Single precision with compensated sums, original basis.
        {"name": "hh2M_sell_f32", "op": "spmv", "matrix": "hh", "n": 2000003, "format": "sell_orig", "dtype": "f32"},
        # A block eigensolver: 16 right-hand sides.
        {"name": "hh1M2_spmm16", "op": "spmm", "matrix": "hh", "n": 1201200, "k": 16, "dtype": "f64"},
        # Forward and backward of one differentiable product.
        {"name": "stencil100_grad", "op": "grad", "matrix": "stencil27", "n": 100, "dtype": "f64"},
        # A training step through twenty products, checkpointed.
        {"name": "stencil100_power20", "op": "power", "matrix": "stencil27", "n": 100, "m": 20, "checkpoint": 5,
         "dtype": "f64"},
        # Many small systems at once: the benchmark's 256 matrices, k in {1, 4, 16}.
        {"name": "batch256_mixed", "op": "batch", "count": 256, "k": "mixed", "dtype": "f64"},
        # Set-up of the tuned storage, paid once per matrix (per time step
        # where the pattern changes).
        {"name": "hh2M_to_sell", "op": "convert", "matrix": "hh", "n": 2000003, "format": "sell_sym", "dtype": "f64"},
        # Set-up of the adjoint.
        {"name": "hh1M2_transpose", "op": "transpose", "matrix": "hh", "n": 1201200, "dtype": "f64"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    dtype = "f32" if rng.random() < 0.25 else "f64"
    op = rng.choice(["spmv", "spmv", "spmv", "spmv", "spmm", "grad", "power", "batch", "convert", "transpose"])
    if op == "spmv":
        matrix = rng.choice(["hh", "hh", "zipf", "laplace"])
        if matrix == "hh":
            return {"op": op, "matrix": matrix, "n": _log_int(rng, 4e3, 5.9e6),
                    "format": rng.choice(["crs", "sell_sym", "sell_orig"]), "dtype": dtype}
        if matrix == "zipf":
            return {"op": op, "matrix": matrix, "n": _log_int(rng, 2e4, 4e6),
                    "format": rng.choice(["crs", "nujds_split"]), "dtype": dtype}
        return {"op": op, "matrix": matrix, "n": _log_int(rng, 32, 1000), "format": rng.choice(["crs", "sell_orig"]),
                "dtype": dtype}
    if op == "spmm":
        return {"op": op, "matrix": rng.choice(["hh", "random"]), "n": _log_int(rng, 4e3, 1.2e6),
                "k": rng.randint(2, 16), "dtype": dtype}
    if op == "grad":
        matrix = rng.choice(["stencil27", "hh"])
        n = _log_int(rng, 12, 100) if matrix == "stencil27" else _log_int(rng, 4e3, 1.2e6)
        return {"op": op, "matrix": matrix, "n": n, "dtype": dtype}
    if op == "power":
        return {"op": op, "matrix": "stencil27", "n": _log_int(rng, 12, 99), "m": rng.randint(4, 20),
                "checkpoint": rng.randint(1, 6), "dtype": dtype}
    if op == "batch":
        return {"op": op, "count": rng.randint(16, 255), "k": rng.choice(["1", "4", "mixed"]), "dtype": dtype}
    if op == "convert":
        return {"op": op, "matrix": rng.choice(["hh", "zipf"]), "n": _log_int(rng, 4e3, 2e6),
                "format": rng.choice(["sell_sym", "sell_orig", "nujds"]), "dtype": dtype}
    return {"op": op, "matrix": rng.choice(["hh", "random", "zipf"]), "n": _log_int(rng, 4e3, 1.2e6), "dtype": dtype}


# --------------------------------------------------------------- inputs --


class _Draws:
    """Random numbers on the GPU from one seed."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed) * 1000003 + 17)

    def rand(self, n):
        return torch.rand(n, generator=self.g, device=DEV, dtype=torch.float64)

    def normal(self, n):
        return torch.randn(n, generator=self.g, device=DEV, dtype=torch.float64)

    def ints(self, lo, hi, n):
        """Integers in [lo, hi]."""
        return torch.randint(lo, hi + 1, (n,), generator=self.g, device=DEV)


def _crs(n, key, val):
    """CRS arrays of a square matrix from its sorted keys row * n + col."""
    row = key // n
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(row, minlength=n), 0, out=row_ptr[1:])
    return row_ptr.int(), (key - row * n).int(), val, n


def _shifted(n, key, d):
    """Keys of the pattern with rows and columns moved by the same distance."""
    s = int(d.ints(0, n - 1, 1))
    return (key // n + s) % n * n + (key % n + s) % n


def _hh(n, d):
    p = _Draws(n)  # the pattern's own draws: every seed gets as many entries
    i = torch.arange(n, device=DEV).repeat_interleave(p.ints(3, 10, n))
    t = i.numel()
    off = torch.tensor(HH_OFFSETS, device=DEV)[p.ints(0, len(HH_OFFSETS) - 1, t)]
    off += torch.where(off >= 256, p.ints(-2, 2, t), 0)
    scattered = i + 1 + (p.rand(t) * (n - 1 - i)).long()
    j = torch.where(p.rand(t) < 0.8, i + off, scattered)
    keep = (j > i) & (j < n)
    upper = torch.unique((i * n + j)[keep])
    del i, j, off, scattered, keep
    v = d.normal(upper.numel())
    diag = torch.arange(n, device=DEV) * (n + 1)
    key = torch.cat([upper, upper % n * n + upper // n, diag])
    val = torch.cat([v, v, d.normal(n)])
    key, order = torch.sort(_shifted(n, key, d))
    return _crs(n, key, val[order])


def _rows(n, lens, p, d):
    i = torch.arange(n, device=DEV).repeat_interleave(lens)
    key = torch.sort(_shifted(n, torch.unique(i * n + p.ints(0, n - 1, i.numel())), d))[0]
    return _crs(n, key, 2 * d.rand(key.numel()) - 1)


def _zipf(n, d):
    p = _Draws(n)
    cdf = torch.cumsum(torch.arange(1, 5001, dtype=torch.float64, device=DEV) ** -2.0, 0)
    lens = 1 + torch.searchsorted(cdf / cdf[-1], p.rand(n), right=True).clamp(max=4999)
    return _rows(n, lens.clamp(max=max(n // 4, 1)), p, d)


def _grid(shape, offsets):
    """Sorted keys of a stencil on a grid (x fastest)."""
    nx, ny, nz = shape
    n = nx * ny * nz
    p = torch.arange(n, device=DEV)
    x, y, z = p % nx, p // nx % ny, p // (nx * ny)
    keys = []
    for a, b, c in offsets:
        ok = (x + a >= 0) & (x + a < nx) & (y + b >= 0) & (y + b < ny) & (z + c >= 0) & (z + c < nz)
        q = p[ok]
        keys.append(q * n + q + a + b * nx + c * nx * ny)
    return n, torch.sort(torch.cat(keys))[0]


_FACES = [(0, 0, 0), (-1, 0, 0), (1, 0, 0), (0, -1, 0), (0, 1, 0)]


def _matrix(name, n, d):
    """(row_ptr, col, val in FP64, n_cols) on the GPU."""
    if name == "hh":
        return _hh(n, d)
    if name == "zipf":
        return _zipf(n, d)
    if name == "random":
        p = _Draws(n)
        return _rows(n, p.ints(5, 30, n), p, d)
    if name == "laplace":
        rows, key = _grid((n, n, 1), _FACES)
        return _crs(rows, key, torch.where(key // rows == key % rows, 4.0, -1.0).double())
    if name == "stencil7":
        shape = (n[0], n[0], n[1])
        rows, key = _grid(shape, _FACES + [(0, 0, -1), (0, 0, 1)])
        return _crs(rows, key, torch.where(key // rows == key % rows, 6.0, -1.0).double())
    rows, key = _grid((n, n, n), [(a, b, c) for c in (-1, 0, 1) for b in (-1, 0, 1) for a in (-1, 0, 1)])
    val = (2 * d.rand(key.numel()) - 1) / 52  # absolute row sums below 1
    return _crs(rows, key, torch.where(key // rows == key % rows, 0.5, val))


def _batch_parts(case, d):
    """The benchmark's batch: sizes log-uniform in [1e3, 2e5], 7-point
    stencils and random rows in turn, with k right-hand sides each."""
    sizes = torch.exp(math.log(1e3) + _Draws(case["count"]).rand(case["count"]) * math.log(200.0))
    sizes = sizes.round().long().tolist()
    for b, n in enumerate(sizes):
        if b % 2:
            A = _matrix("random", n, d)
        else:
            a = max(int(n ** (1 / 3)), 1)
            A = _matrix("stencil7", (a, max(round(n / (a * a)), 1)), d)
        k = (1, 4, 16)[b % 3] if case["k"] == "mixed" else int(case["k"])
        x = 2 * d.rand(A[3] * k) - 1
        yield A, k, x if k == 1 else x.reshape(A[3], k)


def _padded(A, k):
    """Elements of a batch result, with its neighbour on a new 256-byte line."""
    return -(-A[3] * k // 64) * 64


def _inputs(case, seed):
    """Matrix and vectors in the case's precision, vectors in the original basis."""
    d = _Draws(seed)
    dtype = DTYPES[case["dtype"]]
    row_ptr, col, val, n_cols = _matrix(case["matrix"], case["n"], d)
    k = case.get("k", 1)
    x = 2 * d.rand(n_cols * k) - 1
    g = 2 * d.rand(row_ptr.numel() - 1) - 1
    return row_ptr, col, val.to(dtype), n_cols, (x if k == 1 else x.reshape(n_cols, k)).to(dtype), g.to(dtype)


def _convert(M, fmt):
    if fmt in ("nujds", "nujds_split"):
        return M.to_jds("NUJDS", "symmetric", unroll=2)
    return M.to_jds("SELL", "symmetric" if fmt == "sell_sym" else "row_only", window=128, unroll=4)


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        dtype, items = DTYPES[case["dtype"]], []
        parts = list(_batch_parts(case, _Draws(seed)))
        # the results of all matrices in one buffer
        Y = torch.zeros(sum(_padded(A, k) for A, k, _ in parts), dtype=dtype, device=DEV)
        for ((row_ptr, col, val, n_cols), k, x), y in zip(parts, Y.split([_padded(A, k) for A, k, _ in parts])):
            M = CRSMatrix(row_ptr, col, val.to(dtype), n_cols)
            H = M.to_jds("SELL", "row_only", window=1024, unroll=4) if k == 1 else M
            y = y[: n_cols * k]
            items.append((H, x.to(dtype), y if k == 1 else y.view(n_cols, k)))
        return {"op": op, "batch": Batch(items), "Y": Y}
    row_ptr, col, val, n_cols, x, g = _inputs(case, seed)
    if op in ("grad", "power"):
        kept = {"forward": "jds", "adjoint": "jds"} if op == "power" else {}
        return {"op": op, "pattern": Pattern(row_ptr, col, n_cols, val.dtype, **kept), "val": val.requires_grad_(),
                "x": x.requires_grad_(), "g": g, "m": case.get("m"), "checkpoint": case.get("checkpoint")}
    M = CRSMatrix(row_ptr, col, val, n_cols)
    if op in ("convert", "transpose"):
        return {"op": op, "M": M, "format": case.get("format")}
    state = {"op": op, "M": M, "x": x, "original": False}
    fmt = case.get("format", "crs")
    if fmt != "crs":
        state["M"] = J = _convert(M, fmt)
        state["original"] = fmt == "sell_orig"
        if fmt != "sell_orig":  # a solver keeps its vectors in the permuted basis
            state["x"] = J.permute(x)
        if fmt == "nujds_split" and J.n_diag > SPLIT_DEPTH:
            J.split(SPLIT_DEPTH, SPLIT_CHUNK)
    return state


def run(state):
    op = state["op"]
    if op == "spmv":
        return state["M"].spmv_original(state["x"]) if state["original"] else state["M"].spmv(state["x"])
    if op == "spmm":
        return state["M"].spmm(state["x"])
    if op == "batch":
        state["batch"].run()
        return state["Y"]
    if op == "convert":
        J = _convert(state["M"], state["format"])
        layout = [J.jd_ptr] if state["format"] == "nujds" else [J.rlen, J.blk_ptr]
        return [J.val, J.col, J.perm, J.iperm] + layout
    if op == "transpose":
        T = state["M"].transpose()
        return [T.val, T.col, T.row_ptr, T.tmap]
    val, x = state["val"], state["x"]
    if op == "grad":
        y = spmv(state["pattern"], val, x)
    else:
        y = power_apply(state["pattern"], val, x, state["m"], state["checkpoint"])
    dval, dx = torch.autograd.grad(y, (val, x), state["g"])
    if op == "power":
        with torch.no_grad():
            val.sub_(dval, alpha=LEARNING_RATE)
        return [y.detach(), dval, dx, val.detach()]
    return [y.detach(), dval, dx]


# ------------------------------------------------------- work and oracle --


def _size(case):
    """(rows, entries): the recipes' expected entry counts."""
    n, matrix = case["n"], case["matrix"]
    if matrix == "laplace":
        return n * n, 5 * n * n - 4 * n
    if matrix == "stencil27":
        return n ** 3, (3 * n - 2) ** 3
    return n, int(n * {"hh": 13.1, "zipf": 5.52, "random": 17.5}[matrix])


def work(case):
    es = 8 if case["dtype"] == "f64" else 4
    op = case["op"]
    if op == "batch":
        # mean matrix: 199000 / ln 200 rows, half of the matrices with 7 and
        # half with 17.5 entries a row
        n = case["count"] * 199000 / math.log(200)
        k = 7 if case["k"] == "mixed" else int(case["k"])
        return {"bytes": 12.25 * n * (es + 4) + 2 * es * k * n, "flops": 2 * 12.25 * n * k}
    n, nnz = _size(case)
    k = case.get("k", 1)
    matrix, vector = (es + 4) * nnz + 4 * n, es * n
    if op in ("spmv", "spmm"):
        return {"bytes": matrix + 2 * k * vector, "flops": 2 * k * nnz}
    if op == "grad":  # values and pattern once, x and g in, y, dx and dval out
        return {"bytes": matrix + 4 * vector + es * nnz, "flops": 5 * nnz}
    if op == "power":  # every product and its adjoint reads the matrix; values updated
        m = case["m"]
        return {"bytes": 2 * m * (matrix + 2 * vector) + 4 * es * nnz, "flops": 6 * m * nnz}
    if op == "transpose":  # and the entry map
        return {"bytes": 2 * matrix + 4 * nnz, "flops": 0}
    return {"bytes": 2 * matrix + 8 * n, "flops": 0}


def _times(A, rows, x):
    """A x in 64 bits."""
    row_ptr, col, val, _ = A
    p = val.double()
    p = p * x.double()[col.long()] if x.dim() == 1 else p[:, None] * x.double()[col.long()]
    return torch.zeros((row_ptr.numel() - 1,) + x.shape[1:], dtype=torch.float64, device=DEV).index_add_(0, rows, p)


def _row_ids(row_ptr):
    return torch.arange(row_ptr.numel() - 1, device=DEV).repeat_interleave(row_ptr.diff().long())


def _order(row_ptr, window):
    """Stable sort of the rows by decreasing length inside windows."""
    lens = row_ptr.diff().long()
    top = int(lens.max()) + 1
    key = torch.arange(lens.numel(), device=DEV) // window * top + (top - 1 - lens)
    return torch.sort(key, stable=True)[1]


def exact(case, seed):
    op = case["op"]
    if op == "batch":
        out, dtype = [], DTYPES[case["dtype"]]
        for (row_ptr, col, val, n_cols), k, x in _batch_parts(case, _Draws(seed)):
            y = _times((row_ptr, col, val.to(dtype), n_cols), _row_ids(row_ptr), x.to(dtype))
            y = y[_order(row_ptr, 1024)] if k == 1 else y.reshape(-1)
            out.append(torch.nn.functional.pad(y, (0, _padded((0, 0, 0, n_cols), k) - y.numel())))
        return torch.cat(out)
    row_ptr, col, val, n_cols, x, g = _inputs(case, seed)
    A, rows = (row_ptr, col, val, n_cols), _row_ids(row_ptr)
    fmt = case.get("format", "crs")
    window = row_ptr.numel() if fmt.startswith("nujds") else 128
    if op == "spmm":  # column by column: the products of all columns at once need too much memory
        return torch.stack([_times(A, rows, x[:, q].contiguous()) for q in range(x.shape[1])], 1)
    if op == "spmv":
        y = _times(A, rows, x)
        return y if fmt in ("crs", "sell_orig") else y[_order(row_ptr, window)]
    if op == "transpose":
        return [val.double()[torch.sort(col, stable=True)[1]], None, None, None]
    if op == "convert":
        iperm = torch.empty_like(rows[: row_ptr.numel() - 1])
        iperm[_order(row_ptr, window)] = torch.arange(row_ptr.numel() - 1, device=DEV)
        r = iperm[rows]
        slot = torch.arange(col.numel(), device=DEV) - row_ptr.long()[rows]
        block = 32 if fmt != "nujds" else window
        key = (r // block * 8192 + slot) * block + r % block
        return [val.double()[torch.sort(key)[1]]] + [None] * (4 if fmt == "nujds" else 5)
    m = case.get("m", 1)
    xs = [x.double()]
    for _ in range(m):
        xs.append(_times(A, rows, xs[-1]))
    y, gt, c, v = xs.pop(), g.double(), col.long(), val.double()
    dval = torch.zeros_like(v)
    for t in range(m):
        dval += gt[rows] * xs.pop()[c]
        gt = torch.zeros(n_cols, dtype=torch.float64, device=DEV).index_add_(0, c, v * gt[rows])
    return [y, dval, gt] if op == "grad" else [y, dval, gt, v - LEARNING_RATE * dval]
