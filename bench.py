#!/usr/bin/env python
"""Benchmark: FP64 sparse matrix-vector multiplication y = A x on GB300.

Workload (one step = one SpMVM over the whole matrix, the hot path of the
paper's Sect. 2 CRS kernel): the synthetic Holstein-Hubbard-like matrix,
N = 6,000,000 rows, symmetric, banded plus 20% scattered entries, about 13
entries per row (see paper_0910_4836_gb300/synth.py, hh_like).  The matrix
(about 1 GB) is resident in HBM like an operator inside an eigen-solver; x
and y are the step's input and output.

Prints ONE JSON line.  --impl reference times the CPU oracle instead (the
paper's best CPU setting: CRS with an OpenMP static schedule).
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import time

# The CPU oracle's OpenMP threads sit one per core, packed (the paper's
# pinned runs).  Set before any OpenMP runtime in this process starts.
os.environ.setdefault("OMP_PROC_BIND", "close")
os.environ.setdefault("OMP_PLACES", "cores")
# host cores this process may use, read before any OpenMP binding narrows
# the main thread's own mask to one core
AFFINITY_CORES = len(os.sched_getaffinity(0))

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "SpMVM GFlop/s & HBM GB/s vs roofline; batched & fwd+bwd speedup vs plain"
WORKLOAD = ("hh_like N=6,000,000 FP64 SpMVM, fastest of CRS and the JDS family "
            "(symmetric banded + 20% scattered, ~13 nnz/row)")
WORKLOADS = {
    0: "laplace2d 64x64 FP64 SpMVM (5-point, Dirichlet; latency-bound)",
    1: WORKLOAD,
    2: "zipf_rows N=4,000,000 FP64 SpMVM (Zipf(2) row lengths up to 5000, random columns)",
    4: "stencil27 100^3 FP64 SpMVM (27-point, N=1,000,000)",
}
FALLBACK_HBM_GBS = 6800.0


def parse():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=3000)
    p.add_argument("--warmup", type=int, default=5)
    p.add_argument("--impl", default="ours", choices=["ours", "reference"])
    p.add_argument("--config", type=int, default=1, choices=[1, 2, 4])
    p.add_argument("--kernel", default="auto", help="auto, or a name prefix (CRS, JDS, NUJDS, ...)")
    p.add_argument("--no-extras", action="store_true",
                   help="skip the FP32, batched and forward+backward measurements")
    p.add_argument("--cpu-seconds", type=float, default=15.0)
    p.add_argument("--ncu-case", action="store_true",
                   help="no timing: run 3 launches of the --kernel candidate on a 2,000,000-row "
                        "HH-like matrix (larger than L2, small enough for an ncu capture)")
    p.add_argument("--ncu-full", action="store_true",
                   help="with --ncu-case: the full-size workload instead of the 2,000,000-row one")
    p.add_argument("--micro", action="store_true",
                   help="instead of the SpMVM step: the basic gather operations of Sect. 4.1 "
                        "(ADD/SCP over PD, CS, IS, IR; stride sweep; Gaussian stride plane), one JSON line")
    p.add_argument("--analysis", action="store_true",
                   help="instead of the SpMVM step: stride distribution and sectors per warp gather of "
                        "every storage scheme, and block / lanes / window sweeps (Sect. 4.2), one JSON line")
    return p.parse_args()


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return FALLBACK_HBM_GBS, "fallback"


def make_workload(cfg):
    from paper_0910_4836_gb300 import synth as S
    A = S.config(cfg)
    x = S.vector(A.n_cols, cfg)
    return A, x


def algorithmic_bytes(n_rows, n_cols, nnz, vbytes=8):
    # val + col streamed once, row_ptr once, x read at least once, y written once
    return vbytes * nnz + 4 * nnz + 4 * (n_rows + 1) + vbytes * n_cols + vbytes * n_rows


# ------------------------------------------------------------- clocks ------

class ClockSampler:
    """nvidia-smi clock / throttle samples during the timed region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.proc = None
        self.gpu = gpu_index
        self.path = os.path.join("/tmp", f"gbspmv_clocks_{os.getpid()}.csv")

    def __enter__(self):
        try:
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=self.f, stderr=subprocess.DEVNULL)
            time.sleep(0.3)
        except Exception:
            self.proc = None
        return self

    def __exit__(self, *a):
        if self.proc is not None:
            time.sleep(0.2)
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()
            self.f.close()

    def summary(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        rows = []
        with open(self.path) as f:
            for line in f:
                parts = [p.strip() for p in line.split(",")]
                if len(parts) >= 9:
                    rows.append(parts)
        try:
            os.remove(self.path)
        except OSError:
            pass
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i].lower() == "active"})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "samples": len(rows), "reasons": reasons,
                "power_w_max": max((float(r[3]) for r in rows if r[3].replace(".", "").isdigit()),
                                   default=None)}


# ---------------------------------------------------------- distributed ----

def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def max_over_ranks(value: float, device=None) -> float:
    """Largest `value` over all ranks (the job's time is the slowest
    replica's); the identity without a process group."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(value)
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_throughput(units_per_rank: float, world: int, max_ms: float) -> float:
    """Whole-job rate: the units all ranks processed over the slowest time."""
    return world * units_per_rank / (max_ms * 1e-3)


# the functions a step kernel is made of (kernel, its launchers), by scheme
STEP_FUNCTIONS = {"SELL": ("jds.cu", ("store_row_sell(const JdsArgs &a", "sell_walk(const JdsArgs &a)", "sell_kernel(JdsArgs a)", "sell_kernel_f64(JdsArgs a)",
                                     "launch_sell_U(JdsArgs a", "launch_sell(const Mat"))}


def _function_text(src: str, signature: str) -> str:
    """The text of the definition that contains `signature`, from the start
    of its line (attributes such as launch bounds included) and its
    template header, through its closing brace."""
    j = src.index(signature)
    i = src.rfind("\n", 0, j) + 1
    prev = src.rfind("\n", 0, max(i - 1, 0)) + 1
    if src[prev:i].lstrip().startswith("template"):
        i = prev
    j = src.index("{", j)
    depth = 0
    for k in range(j, len(src)):
        depth += {"{": 1, "}": -1}.get(src[k], 0)
        if depth == 0:
            return src[i:k + 1]
    raise ValueError(signature)


def kernel_source_hash(kname: str = "SELL") -> str:
    """Hash of the step kernel's own source (its functions and the
    accumulator header), so that edits elsewhere in the library do not
    invalidate a measurement of it."""
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_0910_4836_gb300", "csrc")
    with open(os.path.join(csrc, "accum.cuh"), "rb") as fh:
        h.update(fh.read())
    fam = STEP_FUNCTIONS.get(kname.split()[0])
    if fam is None:
        with open(os.path.join(csrc, "jds.cu"), "rb") as fh:
            h.update(fh.read())
    else:
        with open(os.path.join(csrc, fam[0])) as fh:
            src = fh.read()
        for sig in fam[1]:
            h.update(_function_text(src, sig).encode())
    return h.hexdigest()[:12]


# DRAM bytes (read + write) per launch of the step kernel on the full
# workload, from one ncu capture (dram__bytes_read.sum + dram__bytes_write.sum,
# a one-pass metric set), keyed by (config, kernel, source hash); a different
# hash means the kernel changed since and traffic is reported null.
NCU_TRAFFIC = {(1, "SELL symmetric w=128 u=4", "fb14ca38e0d1"): 1087956992 + 41890304}


# --------------------------------------------------------------- ours ------

def _timer(dev):
    import torch
    stream = torch.cuda.current_stream(dev)

    def time_launches(fn, reps):
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(reps + 1)]
        torch.cuda.synchronize(dev)
        ev[0].record(stream)
        for i in range(reps):
            fn()
            ev[i + 1].record(stream)
        torch.cuda.synchronize(dev)
        return [ev[i].elapsed_time(ev[i + 1]) for i in range(reps)]

    return time_launches


def jds_method_bytes(A, ptr_entries):
    """Sect. 8(d) method bytes of one JDS-family SpMVM in one basis: val and
    col once (12 B an entry), the format's pointer array (jd_ptr or blk_ptr,
    4 B an entry), x read once and y written once.  The format's own extras
    (SELL's row lengths, the permutation read by a fused basis change) are
    overhead, reported separately."""
    return 12 * A.nnz + 4 * ptr_entries + 8 * A.n_cols + 8 * A.n_rows


class Cand:
    """One timed form of the step: a handle, the vector it reads, the basis
    of x and y, its method bytes and format overhead bytes.  `credited` is
    False for the one form whose output is not A x in a single basis (x in
    the original order, y in the permuted order), kept only for comparison."""

    def __init__(self, name, H, xin, basis, nbytes, overhead=0, how=("fixed",), credited=True):
        self.name, self.H, self.xin, self.basis = name, H, xin, basis
        self.nbytes, self.overhead, self.how, self.credited = nbytes, overhead, how, credited

    def run(self, y):
        from paper_0910_4836_gb300 import _lib as L
        b = L.BASIS_ORIGINAL if self.basis == "original" else L.BASIS_PERMUTED
        self.H.spmv(self.xin, out=y, basis=b)

    def lane_slots(self):
        """FP64 lane-slots of one SELL launch: every block issues 32 lanes
        for each slot of its longest (first) row."""
        H = self.H
        if getattr(H, "fmt", None) != "SELL" or H.rlen is None:
            return None
        import torch
        return int(32 * H.rlen[::32].to(torch.int64).sum().item())


BASIS_LABEL = {
    "original": "original basis: x and y in the user's row order",
    "permuted": "permuted basis (Sect. 2): x and y both in the scheme's row order, y_p = (P A P^T) x_p",
    "mixed": "NOT one basis: x in the original order, y in the permuted row order (uncredited)",
}


def candidates(M, A, x, only=None):
    """Every storage scheme and kernel option on this matrix (the paper's
    serial comparison, Sect. 4.2, on GB300), each in a form whose output is
    A x in one basis: CRS in the original basis; the JDS family with the
    symmetric permutation in the permuted basis (x permuted once, as the
    paper keeps all vectors of a run in that basis); row-only SELL / NUJDS in
    the original basis (y scattered through the permutation inside the
    kernel).  `only`: a name prefix; other schemes are not built."""
    N = A.n_rows
    crs_b = algorithmic_bytes(A.n_rows, A.n_cols, A.nnz)
    out = []
    want = lambda name: only is None or name.startswith(only) or only.startswith(name)
    for l, r in ((4, 4), (8, 2), (16, 2)):
        out.append(Cand(f"CRS vector l{l} r{r}", M, x, "original", crs_b, how=("vector", l, r)))
    for l, r in ((2, 4), (2, 8), (4, 4), (4, 8), (1, 8)):
        out.append(Cand(f"CRS runs l{l} r{r}", M, x, "original", crs_b, how=("runs", l, r)))
    for t in (1024, 2048):
        out.append(Cand(f"CRS tiled {t}", M, x, "original", crs_b, how=("tiled", t)))
    for w, u in ((128, 4), (64, 4), (256, 4), (128, 2)):
        name = f"SELL symmetric w={w} u={u}"
        if want(name):
            G = M.to_jds("SELL", "symmetric", window=w, unroll=u)
            out.append(Cand(name, G, G.permute(x), "permuted", jds_method_bytes(A, G.n_blocks + 1),
                            4 * N))
    for w, u in ((128, 4), (64, 4)):
        name = f"SELL row_only w={w} u={u} original"
        if want(name) or want(f"SELL row_only w={w} u={u} mixed"):
            G = M.to_jds("SELL", "row_only", window=w, unroll=u)
            mb = jds_method_bytes(A, G.n_blocks + 1)
            if want(name):
                out.append(Cand(name, G, x, "original", mb, 8 * N))
            if w == 128 and want(f"SELL row_only w={w} u={u} mixed"):
                out.append(Cand(f"SELL row_only w={w} u={u} mixed", G, x, "mixed", mb, 4 * N,
                                credited=False))
    for w, u in ((64, 2), (128, 4)):
        name = f"PSELL symmetric w={w} u={u}"
        if want(name):
            P = M.to_jds("PSELL", "symmetric", window=w, unroll=u)
            out.append(Cand(name, P, P.permute(x), "permuted", jds_method_bytes(A, P.n_blocks + 1), 4 * N))
    if only is None or any(f.startswith(only) or only.startswith(f)
                           for f in ("JDS", "NUJDS", "NBJDS", "JDS_LITERAL", "RBJDS", "SOJDS")):
        J = M.to_jds("JDS", "symmetric")
        xp = J.permute(x)
        jb = jds_method_bytes(A, J.n_diag + 1)
        for fmt, b, u, r in (("JDS", 0, 0, 1), ("NUJDS", 0, 2, 1), ("NUJDS", 0, 4, 1), ("NUJDS", 0, 8, 1),
                             ("NUJDS", 0, 2, 2), ("NUJDS", 0, 4, 2), ("NUJDS", 0, 2, 4),
                             ("NBJDS", 1024, 0, 1), ("NBJDS", 2048, 0, 1), ("JDS_LITERAL", 0, 0, 1)):
            name = (f"{fmt} symmetric" + (f" b={b}" if b else "") + (f" u={u}" if u else "")
                    + (f" r={r}" if r > 1 else ""))
            out.append(Cand(name, J, xp, "permuted", jb, how=("jds", fmt, b, u, r)))
        for fmt in ("RBJDS", "SOJDS"):
            if want(f"{fmt} symmetric b=1024"):
                R = M.to_jds(fmt, "symmetric", block=1024)
                out.append(Cand(f"{fmt} symmetric b=1024", R, xp, "permuted",
                                jb + 4 * (R.n_blocks + 1)))
    if want("NUJDS row_only u=2 original"):
        Jr = M.to_jds("NUJDS", "row_only", unroll=2)
        out.append(Cand("NUJDS row_only u=2 original", Jr, x, "original", jds_method_bytes(A, Jr.n_diag + 1),
                        4 * N))
    return out


def configure(H, how):
    if how[0] in ("vector", "runs"):
        H.set_kernel(how[0], lanes=how[1], rows_per_warp=how[2])
    elif how[0] == "tiled":
        H.prepare_tiled(how[1])
    elif how[0] == "jds":
        H.set_format(how[1], block=how[2], unroll=how[3])
        H.set_kernel("vector", rows_per_warp=how[4])


def fp64_rate(dev, time_launches):
    """The FP64 FMA issue rate of this GPU (gbsp_fma_chain): every SM full
    (8 CTAs of 256 threads), 8 independent FMA chains a thread, median of 5
    launches; again with half the lanes of every warp idle, which takes the
    same time when an idle lane costs what a busy one does."""
    import torch
    from paper_0910_4836_gb300.gather import FmaChain
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    out = {"sms": sms, "threads": sms * 2048, "iters": 1024}
    for active in (32, 16):
        f = FmaChain(sms * 2048, active_lanes=active, iters=1024, device=dev)
        f()
        t = statistics.median(time_launches(f, 5))
        out[f"tflops_{active}_lanes"] = round(f.flops / (t * 1e-3) / 1e12, 4)
        out[f"ms_{active}_lanes"] = round(t, 4)
        # every warp-wide FMA instruction, idle lanes counted as busy
        out[f"lane_slot_tflops_{active}_lanes"] = round(16.0 * 1024 * sms * 2048 / (t * 1e-3) / 1e12, 4)
        del f
    out["tflops"] = out["tflops_32_lanes"]
    return out


def cold_times(fn, dev, reps=20):
    """Times of `fn` with L2 flushed before each launch (a 512 MB write,
    four times the 129 MB L2), CUDA events around the launch only."""
    import torch
    stream = torch.cuda.current_stream(dev)
    flush = torch.empty(64 * 2 ** 20, dtype=torch.float64, device=dev)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    out = []
    for _ in range(reps):
        flush.fill_(1.0)
        e0.record(stream)
        fn()
        e1.record(stream)
        e1.synchronize()
        out.append(e0.elapsed_time(e1))
    del flush
    return out


def run_ours(args):
    import torch
    world, rank, local = dist_env()
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    dev = torch.device("cuda", local if world > 1 else 0)
    torch.cuda.set_device(dev)

    import paper_0910_4836_gb300 as g
    from paper_0910_4836_gb300 import CRSMatrix
    g.build()
    time_launches = _timer(dev)

    A, x_host = make_workload(args.config)
    M = CRSMatrix.from_host(A, device=dev, dtype=torch.float64)
    x = torch.as_tensor(x_host).to(dev)
    y = torch.empty(A.n_rows, dtype=torch.float64, device=dev)
    peak, peak_kind = peaks()
    fp64 = fp64_rate(dev, time_launches)

    # every form timed (median of 10 launches); the fastest credited one is
    # the step
    table, best = {}, None
    for c in candidates(M, A, x, None if args.kernel == "auto" else args.kernel):
        if args.kernel != "auto" and not c.name.startswith(args.kernel):
            continue
        configure(c.H, c.how)
        t = statistics.median(time_launches(lambda: c.run(y), 10))
        table[c.name] = {"gflops": round(2.0 * A.nnz / (t * 1e-3) / 1e9, 1),
                         "gbs": round(c.nbytes / (t * 1e-3) / 1e9, 1), "ms": round(t, 4),
                         "frac": round(c.nbytes / (t * 1e-3) / 1e9 / peak, 3), "basis": c.basis}
        if not c.credited:
            table[c.name]["credited"] = False
            continue
        # a later scheme replaces the choice only when more than 1% faster,
        # so near-ties keep the earlier (listed first) scheme from run to run
        if best is None or t < 0.99 * best[0]:
            best = (t, c)
    _, step_c = best
    kname, H, xin, alg = step_c.name, step_c.H, step_c.xin, step_c.nbytes
    configure(H, step_c.how)

    def step():
        step_c.run(y)

    for _ in range(max(args.warmup, 3)):
        step()
    torch.cuda.synchronize(dev)
    if world > 1:
        torch.distributed.barrier()
    with ClockSampler(torch.cuda.current_device() if world == 1 else local) as clk:
        times = time_launches(step, args.steps)
        torch.cuda.synchronize(dev)
    if world > 1:
        torch.distributed.barrier()
    total_ms = max_over_ranks(sum(times), dev)
    ms = total_ms / args.steps
    flops = 2.0 * A.nnz
    gflops = job_throughput(flops, world, ms) / 1e9
    gbs = alg / (ms * 1e-3) / 1e9
    h = kernel_source_hash(kname)
    traffic = NCU_TRAFFIC.get((args.config, kname, h))
    cold_ms = statistics.median(cold_times(step, dev))
    slots = step_c.lane_slots()

    # end to end through the public API, in the original basis so that the
    # host gets y = A x in its own row order: every step is one C-ABI call
    # with host vectors (gbsp_spmv_host), which copies x in from pinned host
    # memory, runs the product (row-only SELL, y scattered through the
    # permutation in the kernel) and copies y back to pinned host memory, in
    # order on its stream.  Steps go round-robin over four streams, each with
    # its own device stages and host output, so copies in both directions and
    # the products overlap.
    from paper_0910_4836_gb300 import _lib as L
    if step_c.basis == "original":
        He, e2e_kernel = H, kname
    else:
        He, e2e_kernel = M.to_jds("SELL", "row_only", window=128, unroll=4), "SELL row_only w=128 u=4 original"
    nstr = 4
    xh = x.detach().cpu().pin_memory()
    yh = [torch.empty(A.n_rows, dtype=torch.float64).pin_memory() for _ in range(nstr)]
    stages = [He.host_stage() for _ in range(nstr)]
    streams = [torch.cuda.Stream(dev) for _ in range(nstr)]
    main = torch.cuda.current_stream(dev)

    def e2e_steps(n):
        for i in range(n):
            b = i % nstr
            He.spmv_host(xh, out=yh[b], stage=stages[b], stream=streams[b], basis=L.BASIS_ORIGINAL)

    def fenced(n):
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record(main)
        for st in streams:
            st.wait_event(t0)
        e2e_steps(n)
        for st in streams:
            main.wait_stream(st)
        t1.record(main)
        return t0, t1

    fenced(4)
    torch.cuda.synchronize(dev)
    e2e_n = 50
    t_start, t_end = fenced(e2e_n)
    torch.cuda.synchronize(dev)
    e2e_ms = t_start.elapsed_time(t_end) / e2e_n
    del He, stages

    result = None
    if rank == 0:
        rate = fp64["tflops"] * 1e12
        result = {
            "metric": METRIC, "value": round(gflops, 2), "unit": "GFlop/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(ms, 5),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic (seeded SplitMix64; stand-in for the paper's Holstein-Hubbard matrix)",
            "hbm_gbs": round(gbs, 1),
            "config": {"workload": WORKLOADS.get(args.config, WORKLOAD), "config_index": args.config, "n_rows": A.n_rows,
                       "nnz": A.nnz, "kernel": kname, "vectors": BASIS_LABEL[step_c.basis],
                       "l2": "inputs larger than L2 (matrix ~1 GB), no flush between timed steps; "
                             "roofline.cold_ms flushes L2 before each launch",
                       "parallelism": f"replicas x{world}"},
            "roofline": {"bound": "hbm", "achieved": round(gbs, 1), "peak": peak, "unit": "GB/s",
                         "frac": round(gbs / peak, 4), "traffic": traffic,
                         "frac_of_8tbs_spec": round(gbs / 8000.0, 4),
                         "algorithmic_bytes": alg,
                         "algorithmic_bytes_formula": "12 nnz + 4 (pointer entries) + 8 N_c + 8 N",
                         "format_overhead_bytes": step_c.overhead,
                         "format_overhead": ("SELL row lengths 4N" if kname.startswith("SELL") else
                                             "none" if kname.startswith("CRS") else "JDS-family extras") +
                                            (" + permutation 4N read by the fused basis change"
                                             if step_c.basis == "original" and not kname.startswith("CRS") else ""),
                         "peak_source": f"{peak_kind} hbm_gbs (burst)",
                         "kernel_source_hash": h,
                         "cold_ms": round(cold_ms, 5),
                         "cold_frac": round(alg / (cold_ms * 1e-3) / 1e9 / peak, 4),
                         "fp64_fma_tflops": fp64["tflops"],
                         "fp64_floor_us": round(2.0 * A.nnz / rate * 1e6, 1),
                         "fp64_lane_slots": slots,
                         "fp64_slot_floor_us": None if slots is None else round(2.0 * slots / rate * 1e6, 1),
                         "hbm_floor_us": round(alg / (peak * 1e9) * 1e6, 1)},
            "fp64_rate": fp64,
            "e2e": {"value": round(world * flops / (e2e_ms * 1e-3) / 1e9, 2), "unit": "GFlop/s",
                    "h2d_bytes_per_step": 8 * A.n_cols, "d2h_bytes_per_step": 8 * A.n_rows,
                    "ms_per_step": round(e2e_ms, 4), "kernel": e2e_kernel,
                    "vectors": BASIS_LABEL["original"],
                    "how": "one gbsp_spmv_host call per step (pinned host x in, product, pinned host y out, "
                           "in order on its stream); steps round-robin over four streams and stage sets"},
            "gpu_launches": args.steps * launches_per_step(kname, H),
            "clocks": clk.summary(),
            "formats": table,
        }
        fp32_dev = None
        if not args.no_extras:
            result["fp32"], fp32_dev = fp32_numbers(M, A, x, y, dev, time_launches, table[kname]["ms"])
            torch.cuda.empty_cache()
            result["symmetric"] = symmetric_numbers(M, A, x, dev, time_launches, table[kname]["ms"])
            del table
            torch.cuda.empty_cache()
            result["spmm_adjoint"] = spmm_adjoint_numbers(M, A, x, dev, time_launches, peak)
            torch.cuda.empty_cache()
            result["batched"] = batched_speedups(dev, time_launches)
            torch.cuda.empty_cache()
            result["fwd_bwd"] = fwd_bwd_speedup(dev, time_launches)
            torch.cuda.empty_cache()
            result["zipf_rows"] = zipf_numbers(dev, time_launches, peak)
            torch.cuda.empty_cache()
            result["hybrid_dia"] = hybrid_numbers(dev, time_launches, peak)
            torch.cuda.empty_cache()
            result["laplace_64x64"] = small_numbers(dev, time_launches)
        result["cpu_baseline"] = cpu_baseline(A, x_host, args.cpu_seconds, fp32_dev)
        if "fp32" in result:
            result["fp32"]["per_config"] = result["cpu_baseline"].pop("fp32_error_vs_oracle")
    if world > 1:
        torch.distributed.barrier()
        torch.distributed.destroy_process_group()
    return result


def launches_per_step(kname, H):
    if kname.startswith("JDS_LITERAL"):
        return int(H.n_diag) + 1  # one zeroing launch and one launch per diagonal
    return 1



# ------------------------------------------------------------- extras ------

def fp32_numbers(M, A, x, y64, dev, time_launches, ms64):
    """FP32 values with compensated (Dot2) row sums on the same matrix: the
    speed of each FP32 kernel against the FP64 step.  Also returns, for the
    CPU leg, the FP32 products (compensated and plain) of every workload,
    whose errors against the FP64 oracle that leg states."""
    import torch
    from paper_0910_4836_gb300 import CRSMatrix
    M32 = CRSMatrix(M.row_ptr, M.col, M.val.float(), A.n_cols)
    M32.set_kernel("vector", compensated=True)
    x32 = x.float()
    y32 = torch.empty(A.n_rows, dtype=torch.float32, device=dev)
    J32 = M32.to_jds("NUJDS", "symmetric", unroll=4)
    xp32 = J32.permute(x32)
    G32 = M32.to_jds("SELL", "symmetric", window=128, unroll=4)
    G32o = M32.to_jds("SELL", "row_only", window=128, unroll=4)
    xs32 = G32.permute(x32)
    res = {}
    opts = [("CRS vector l4 r4", M32, x32, lambda: M32.set_kernel("vector", lanes=4, rows_per_warp=4), 0),
            ("CRS tiled 1024", M32, x32, lambda: M32.prepare_tiled(1024), 0),
            ("NUJDS symmetric u=4", J32, xp32, lambda: None, 0),
            ("SELL symmetric w=128 u=4", G32, xs32, lambda: None, 0),
            ("SELL row_only w=128 u=4 original", G32o, x32, lambda: None, 1)]
    best = None
    for name, H, xin, conf, basis in opts:
        conf()
        t = statistics.median(time_launches(lambda: H.spmv(xin, out=y32, basis=basis), 10))
        res[name] = {"gflops": round(2.0 * A.nnz / (t * 1e-3) / 1e9, 1), "ms": round(t, 4),
                     "gbs": round((8 * A.nnz + 4 * (A.n_rows + 1) + 4 * (A.n_rows + A.n_cols))
                                  / (t * 1e-3) / 1e9, 1)}
        if best is None or t < best[0]:
            best = (t, name)
    del M32, J32, G32, G32o
    torch.cuda.empty_cache()
    out = {"best": best[1], "speedup_vs_fp64": round(ms64 / best[0], 3), "kernels": res,
           "note": "error of the FP32 product (FP32 values and vector) against the FP64 oracle, max over rows "
                   "of |y32 - y| / sum|a||x|; 'dot2_bound_ok' checks the compensated sums against the Dot2 "
                   "bound relative to the exact product of the FP32-rounded data"}
    return out, fp32_products(dev)


def fp32_products(dev):
    """FP32 products of each workload on the GPU (FP32 values and vector; CRS
    with compensated and with plain row sums), copied to the host for the
    oracle comparison: the Laplacian, the HH-like matrix, the Zipf rows and
    the 27-point stencil."""
    import torch
    from paper_0910_4836_gb300 import CRSMatrix, synth as S
    out = {}
    for i, name in ((0, "laplace_64x64"), (1, "hh_like_6M"), (2, "zipf_rows_4M"), (4, "stencil27_100^3")):
        A = S.config(i)
        xh = S.vector(A.n_cols, i)
        M32 = CRSMatrix.from_host(A, device=dev, dtype=torch.float32)
        x32 = torch.as_tensor(xh).to(dev).float()
        ys = {}
        for comp in (True, False):
            M32.set_kernel("vector", lanes=4, rows_per_warp=4, compensated=comp)
            ys["compensated" if comp else "plain"] = M32.spmv(x32).cpu().numpy()
        out[name] = (A, xh, ys)
        del M32
        torch.cuda.empty_cache()
    return out


def fp32_error_vs_oracle(products):
    """For each workload: max over rows of |y32 - y_oracle| / sum|a||x|,
    y_oracle the accurate FP64 oracle product of the FP64 data; and whether
    the compensated sums meet the Dot2 bound against the exact product of
    the FP32-rounded data."""
    import oracle as O
    from paper_0910_4836_gb300 import synth as S
    out = {}
    for name, (A, xh, ys) in products.items():
        ref, s = O.crs_spmv_exact(A, xh)
        den = np.maximum(s, 1e-300)
        row = {k: float(np.max(np.abs(v.astype(np.float64) - ref) / den)) for k, v in ys.items()}
        A32 = S.CRS(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val.astype(np.float32).astype(np.float64), A.name)
        r32, s32 = O.crs_spmv_exact(A32, xh.astype(np.float32).astype(np.float64))
        n = np.maximum(A.row_lengths(), 1).astype(np.float64) + 6.0
        u = 2.0 ** -24
        gam = n * u / (1 - n * u)
        bound = 2 * u * np.abs(r32) + (gam * gam + n * u * u) * s32
        row["dot2_bound_ok"] = bool(np.all(np.abs(ys["compensated"].astype(np.float64) - r32) <= bound))
        out[name] = row
    return out


def spmm_adjoint_numbers(M, A, x, dev, time_launches, peak):
    """The SpMM, adjoint and dval rows on the HH-like matrix, each against
    its own algorithmic bytes and the HBM peak: Y = A X for k = 4 and 16
    (CRS and SELL), A^T g through the transposed CRS and through a NUJDS of
    A^T, and dval_k = g[row_k] x[col_k]."""
    import torch
    N, Nc, nnz = A.n_rows, A.n_cols, A.nnz
    out = {}

    def row(t_ms, nbytes, flops):
        return {"ms": round(t_ms, 4), "gflops": round(flops / (t_ms * 1e-3) / 1e9, 1),
                "gbs": round(nbytes / (t_ms * 1e-3) / 1e9, 1),
                "frac": round(nbytes / (t_ms * 1e-3) / 1e9 / peak, 3)}

    M.set_kernel("vector", lanes=4, rows_per_warp=4)
    G = M.to_jds("SELL", "row_only", window=128, unroll=4)
    for k in (4, 16):
        X = torch.rand(Nc, k, dtype=torch.float64, device=dev)
        Y = torch.empty(N, k, dtype=torch.float64, device=dev)
        nb = 12 * nnz + 4 * (N + 1) + 8 * k * (Nc + N)
        for name, fn in (("CRS", lambda: M.spmm(X, out=Y)),
                         ("SELL row_only w=128 original", lambda: G.spmm(X, out=Y, basis=1))):
            t = statistics.median(time_launches(fn, 10))
            out[f"spmm k={k} {name}"] = row(t, nb, 2.0 * nnz * k)
        del X, Y
    del G
    torch.cuda.empty_cache()
    T = M.transpose()
    g = torch.rand(N, dtype=torch.float64, device=dev)
    z = torch.empty(Nc, dtype=torch.float64, device=dev)
    ab = 12 * nnz + 4 * (Nc + 1) + 8 * N + 8 * Nc
    t = statistics.median(time_launches(lambda: M.spmv(g, out=z, transpose=True), 10))
    out["adjoint A^T g, transposed CRS"] = row(t, ab, 2.0 * nnz)
    JT = T.to_jds("NUJDS", "row_only", unroll=2)
    t = statistics.median(time_launches(lambda: JT.spmv(g, out=z, basis=1), 10))
    out["adjoint A^T g, NUJDS of A^T, original basis"] = row(t, 12 * nnz + 4 * (JT.n_diag + 1) + 16 * Nc, 2.0 * nnz)
    del JT
    d = torch.empty(nnz, dtype=torch.float64, device=dev)
    db = 8 * nnz + 4 * nnz + 4 * (N + 1) + 8 * N + 8 * Nc
    t = statistics.median(time_launches(lambda: M.dval(g, x, out=d), 10))
    out["dval"] = row(t, db, 1.0 * nnz)
    out["bytes"] = {"spmm": "12 nnz + 4(N+1) + 8k(N_c+N)", "adjoint": "12 nnz + 4(N_c+1) + 8N + 8N_c",
                    "dval": "8 nnz written + 4 nnz col + 4(N+1) + 8N + 8N_c"}
    return out


def symmetric_numbers(M, A, x, dev, time_launches, ms_full):
    """The product from the upper triangle only (FP64 atomic scatter of the
    transposed half) on the same matrix: its time against the full-storage
    step, and the entries it reads."""
    import torch
    U = M.upper()
    y = torch.zeros(A.n_rows, dtype=torch.float64, device=dev)
    out = {"nnz_upper": U.nnz, "nnz_full": A.nnz, "full_step_ms": ms_full}
    for name, H in (("CRS upper", U), ("SELL upper row_only w=128 u=4", U.to_jds("SELL", "row_only", window=128,
                                                                                 unroll=4))):
        t = statistics.median(time_launches(lambda: H.spmv_symmetric(x, out=y), 10))
        out[name] = {"ms": round(t, 4), "gflops": round(2.0 * A.nnz / (t * 1e-3) / 1e9, 1),
                     "speedup_vs_full": round(ms_full / t, 3)}
    return out


def hybrid_numbers(dev, time_launches, peak):
    """The DIA + remainder hybrid on the second HH stand-in (60% of the
    entries on twelve dense outer diagonals, as Sect. 4.2 describes the real
    matrix), against SELL and CRS on the same matrix."""
    import torch
    from paper_0910_4836_gb300 import CRSMatrix, HybridMatrix, synth as S
    A = S.hh_diagonals(6_000_000, 5)
    M = CRSMatrix.from_host(A, device=dev)
    x = torch.as_tensor(S.vector(A.n_cols, 5)).to(dev)
    y = torch.empty(A.n_rows, dtype=torch.float64, device=dev)
    crs_b = algorithmic_bytes(A.n_rows, A.n_cols, A.nnz)
    out = {"workload": "hh_diagonals N=6,000,000 (12 dense outer diagonals + band of 400)", "nnz": A.nnz,
           "kernels": {}}

    def rec(name, fn, nbytes):
        t = statistics.median(time_launches(fn, 10))
        out["kernels"][name] = {"ms": round(t, 4), "gflops": round(2.0 * A.nnz / (t * 1e-3) / 1e9, 1),
                                "gbs": round(nbytes / (t * 1e-3) / 1e9, 1),
                                "frac": round(nbytes / (t * 1e-3) / 1e9 / peak, 3)}

    M.set_kernel("vector", lanes=4, rows_per_warp=4)
    rec("CRS vector l4 r4", lambda: M.spmv(x, out=y), crs_b)
    G = M.to_jds("SELL", "row_only", window=128, unroll=4)
    rec("SELL row_only w=128 u=4 original", lambda: G.spmv(x, out=y, basis=1),
        12 * A.nnz + 4 * (G.n_blocks + 1) + 20 * A.n_rows)
    del G
    for rem in ("SELL", "CRS"):
        H = HybridMatrix(M, 16, 2.0 / 3.0, remainder=rem, window=128, unroll=4)
        nd = len(H.offsets_host)
        hb = 8 * nd * A.n_rows + 12 * H.nnz_rem + 4 * (A.n_rows + 1) + 16 * A.n_rows
        rec(f"hybrid DIA({nd}) + {rem}", lambda: H.spmv(x, out=y), hb)
        out["dia_diagonals"], out["nnz_dia"] = nd, H.nnz_dia
        del H
    return out


def small_numbers(dev, time_launches):
    """The 64x64 Laplacian (N=4096, fits in L2): latency-bound, so the figures
    are microseconds per SpMVM, eager (one launch each) and as one replay of
    a CUDA graph holding 100 SpMVMs."""
    import torch
    from paper_0910_4836_gb300 import CRSMatrix, synth as S
    A = S.config(0)
    M = CRSMatrix.from_host(A, device=dev)
    x = torch.as_tensor(S.vector(A.n_cols, 0)).to(dev)
    out = {"n_rows": A.n_rows, "nnz": A.nnz}
    for name, H, xin in (("CRS vector", M, x),
                         ("SELL row_only w=128 u=4 original", M.to_jds("SELL", "row_only", window=128, unroll=4), x),
                         ("NUJDS row_only u=2 original", M.to_jds("NUJDS", "row_only", unroll=2), x)):
        if name.startswith("CRS"):
            H.autotune()
        y = torch.empty(A.n_rows, dtype=torch.float64, device=dev)
        b = 0 if name.startswith("CRS") else 1
        eager = statistics.median(time_launches(lambda: H.spmv(xin, out=y, basis=b), 200))
        s = torch.cuda.Stream(dev)
        s.wait_stream(torch.cuda.current_stream(dev))
        with torch.cuda.stream(s):
            H.spmv(xin, out=y, basis=b)
        torch.cuda.current_stream(dev).wait_stream(s)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for _ in range(100):
                H.spmv(xin, out=y, basis=b)
        replay = statistics.median(time_launches(g.replay, 20)) / 100
        out[name] = {"eager_us": round(eager * 1e3, 2), "graph_us": round(replay * 1e3, 2)}
    return out


def zipf_candidates(M, A, x, y):
    """(name, launch, method bytes) of the Zipf-rows forms: CRS vector and
    tiled, and NUJDS with the deep-diagonal split in the permuted basis
    (columns are uniform random, so the symmetric renumbering costs no
    locality; x is permuted once)."""
    crs_b = algorithmic_bytes(A.n_rows, A.n_cols, A.nnz)
    runs = []
    M.set_kernel("vector", lanes=4, rows_per_warp=4)
    runs.append(("CRS vector l4 r4", lambda: M.spmv(x, out=y), crs_b))
    from paper_0910_4836_gb300 import CRSMatrix
    for l, r in ((2, 8), (4, 4)):
        Mr = CRSMatrix(M.row_ptr, M.col, M.val, A.n_cols)
        Mr.set_kernel("runs", lanes=l, rows_per_warp=r)
        runs.append((f"CRS runs l{l} r{r}", lambda Mr=Mr: Mr.spmv(x, out=y), crs_b))
    M2 = CRSMatrix(M.row_ptr, M.col, M.val, A.n_cols)
    M2.prepare_tiled(1024)
    runs.append(("CRS tiled 1024", lambda: M2.spmv(x, out=y), crs_b))
    J = M.to_jds("NUJDS", "symmetric", unroll=2)
    xp = J.permute(x)
    J.split(16, 64)
    runs.append(("NUJDS symmetric u=2 split 16/64", lambda: J.spmv(xp, out=y), jds_method_bytes(A, J.n_diag + 1)))
    return runs


def zipf_numbers(dev, time_launches, peak):
    """The irregular workload (N = 4e6, Zipf(2) row lengths up to 5000,
    random columns): FP64 SpMVM in the candidate schemes; JDS needs the
    deep-diagonal split, since a few rows have thousands of entries."""
    import torch
    from paper_0910_4836_gb300 import CRSMatrix, synth as S
    A = S.config(2)
    M = CRSMatrix.from_host(A, device=dev)
    x = torch.as_tensor(S.vector(A.n_cols, 2)).to(dev)
    y = torch.empty(A.n_rows, dtype=torch.float64, device=dev)
    out = {"n_rows": A.n_rows, "nnz": A.nnz, "max_row": int(A.row_lengths().max())}
    table, best = {}, None
    for name, fn, nbytes in zipf_candidates(M, A, x, y):
        t = statistics.median(time_launches(fn, 10))
        table[name] = {"gflops": round(2.0 * A.nnz / (t * 1e-3) / 1e9, 1), "ms": round(t, 4),
                       "gbs": round(nbytes / (t * 1e-3) / 1e9, 1),
                       "frac": round(nbytes / (t * 1e-3) / 1e9 / peak, 3)}
        if best is None or t < best[0]:
            best = (t, name)
    out["kernels"] = table
    out["best"] = best[1]
    return out


def batched_speedups(dev, time_launches):
    """256 uneven matrices (half 7-point stencils, half random rows) in one
    persistent launch replayed from a CUDA graph, against the plain path:
    one CRS launch per matrix and right-hand side, launched eagerly (host
    overhead included, as a plain caller pays it) and replayed from a graph
    (GPU side only)."""
    import torch
    from paper_0910_4836_gb300 import Batch, CRSMatrix, synth as S
    mats = S.batch_set(256, 3)
    out = {"matrices": len(mats), "rows": int(sum(m.n_rows for m in mats)),
           "nnz": int(sum(m.nnz for m in mats))}
    for dtype, kmode in ((torch.float64, "1"), (torch.float64, "16"), (torch.float64, "mixed"),
                         (torch.float32, "mixed")):
        ks = S.batch_k(len(mats), kmode)
        bt, handles, Xs, Ys = Batch.autotuned(mats, ks, dtype, device=dev, chunk=16384)
        for X in Xs:
            X.uniform_(-1, 1)
        g = bt.graph()
        t_batch = statistics.median(time_launches(g.replay, 20))
        t_cold = statistics.median(cold_times(g.replay, dev, 10))
        plain = [CRSMatrix(h.row_ptr, h.col, h.val, h.n_cols) if isinstance(h, CRSMatrix)
                 else CRSMatrix.from_host(m, device=dev, dtype=dtype) for h, m in zip(handles, mats)]
        for P in plain:
            if dtype == torch.float32:
                P.set_kernel("vector", compensated=True)
        cols = [[torch.empty(m.n_cols, dtype=dtype, device=dev).uniform_(-1, 1) for _ in range(k)]
                for m, k in zip(mats, ks)]
        outs = [torch.empty(m.n_rows, dtype=dtype, device=dev) for m in mats]

        def plain_run():
            for P, cs, o in zip(plain, cols, outs):
                for c in cs:
                    P.spmv(c, out=o)

        t_plain = statistics.median(time_launches(plain_run, 5))
        # the same plain launches replayed from one CUDA graph: no host
        # overhead per launch, so what is left is the GPU side of the gain
        # (one persistent launch balanced over the CTAs against one small
        # launch per matrix and right-hand side)
        plain_run()
        torch.cuda.synchronize(dev)
        pg = torch.cuda.CUDAGraph()
        with torch.cuda.graph(pg):
            plain_run()
        t_plain_graph = statistics.median(time_launches(pg.replay, 10))
        flops = sum(2.0 * m.nnz * k for m, k in zip(mats, ks))
        nw, grid = bt.info()
        out[f"{'f64' if dtype == torch.float64 else 'f32'}_k{kmode}"] = {
            "batched_ms": round(t_batch, 4), "batched_cold_ms": round(t_cold, 4), "plain_ms": round(t_plain, 4),
            "speedup": round(t_plain / t_batch, 2), "batched_gflops": round(flops / (t_batch * 1e-3) / 1e9, 1),
            "plain_graph_ms": round(t_plain_graph, 4), "speedup_vs_plain_graph": round(t_plain_graph / t_batch, 2),
            "launches_plain": int(sum(ks)), "work_items": nw, "ctas": grid,
            "jds_items": sum(1 for h in handles if not isinstance(h, CRSMatrix))}
        del bt, handles, Xs, Ys, plain, cols, outs, g, pg
        torch.cuda.empty_cache()
    return out


def fwd_bwd_speedup(dev, time_launches):
    """loss = ||A^20 x||^2 on the 27-point stencil, 100^3: forward and
    backward, plain (all 20 activations stored, one dval launch per step,
    CRS of A^T) against tuned (autotuned forward and adjoint handles,
    checkpoint every 5 steps, fused multi-step dval).  Both sides run on
    fixed values; the same pair is also timed with a value update before
    every pass (new values: the tuned handles re-gather theirs, the plain
    CRS of A^T its own), as in a training step."""
    import torch
    from paper_0910_4836_gb300 import synth as S
    from paper_0910_4836_gb300.autograd import Pattern, power_apply
    A = S.stencil27(100, 4)
    m = 20
    res = {"n_rows": A.n_rows, "nnz": A.nnz, "m": m}
    for dtype in (torch.float64, torch.float32):
        # plain: default CRS kernels, explicit transposed CRS
        p = Pattern.from_host(A, device=dev, dtype=dtype)
        # tuned: autotuned forward and adjoint kernels (CRS or JDS, either side)
        pt = Pattern.from_host(A, device=dev, dtype=dtype, forward="auto", adjoint="auto")
        val = torch.as_tensor(A.val).to(device=dev, dtype=dtype)
        x0 = torch.as_tensor(S.vector(A.n_cols, 4)).to(device=dev, dtype=dtype)
        M = p.bind(val)
        p.adjoint_op(val)  # build the transposed structure once
        AT = p.AT
        vparam = val.clone().requires_grad_(True)
        pt.forward_op(vparam)
        pt.adjoint_op(vparam)

        def plain(update=False):
            if update:
                M.refresh_transpose_values()
            xs = [x0]
            for _ in range(m):
                xs.append(M.spmv(xs[-1]))
            g = 2 * xs[-1]
            dval = torch.zeros(A.nnz, dtype=dtype, device=dev)
            for t in range(m, 0, -1):
                M.dval(g, xs[t - 1], out=dval, accumulate=True)
                g = AT.spmv(g)
            return dval, g

        def tuned(c=5, update=False):
            # update: a new values tensor, so the tuned handles re-gather
            # their values through the value maps (as after an optimiser step)
            v = val.clone().requires_grad_(True) if update else vparam
            v.grad = None
            xx = x0.clone().requires_grad_(True)
            y = power_apply(pt, v, xx, m, checkpoint=c)
            (y * y).sum().backward()
            return v.grad, xx.grad

        for _ in range(2):
            plain(), tuned(), tuned(1), plain(True), tuned(update=True)
        tp = statistics.median(time_launches(plain, 5))
        tt = statistics.median(time_launches(tuned, 5))
        t1 = statistics.median(time_launches(lambda: tuned(1), 5))
        tpu = statistics.median(time_launches(lambda: plain(True), 5))
        ttu = statistics.median(time_launches(lambda: tuned(update=True), 5))
        key = "f64" if dtype == torch.float64 else "f32"
        res[key] = {"plain_ms": round(tp, 3), "tuned_ms": round(tt, 3), "speedup": round(tp / tt, 3),
                    "vectors_stored_plain": m + 1, "vectors_stored_tuned": m // 5 + 5,
                    "tuned_forward": getattr(pt.F, "fmt", "CRS"), "tuned_adjoint": getattr(pt._adj, "fmt", "CRS"),
                    "checkpoint": 5, "values": "fixed",
                    "tuned_all_stored": {"checkpoint": 1, "ms": round(t1, 3), "speedup": round(tp / t1, 3),
                                         "vectors_stored": m + 1},
                    "with_value_update": {"plain_ms": round(tpu, 3), "tuned_ms": round(ttu, 3),
                                          "speedup": round(tpu / ttu, 3),
                                          "what": "new values before every pass: the tuned handles re-gather "
                                                  "theirs, the plain transposed CRS its own"}}
    return res


# ------------------------------------------------------------ CPU side -----

def host_copy_gbs(nbytes=1 << 30, reps=5):
    """STREAM-style copy bandwidth of the host (torch CPU copy, all its
    threads), read + write bytes per second: the CPU side's own roofline."""
    import torch
    src = torch.ones(nbytes // 8, dtype=torch.float64)
    dst = torch.empty_like(src)
    dst.copy_(src)
    best = None
    for _ in range(reps):
        t0 = time.perf_counter()
        dst.copy_(src)
        el = time.perf_counter() - t0
        best = el if best is None else min(best, el)
    return round(2 * nbytes / best / 1e9, 1)


def cpu_baseline(A, x, seconds, fp32_products=None):
    """The oracle on the host cores: its OpenMP static-schedule CRS loop (the
    paper's best parallel setting) on the full matrix, repeated for about
    `seconds`; the serial literal CRS and JDS loops on one core, once each;
    the host copy bandwidth; and, given the GPU's FP32 products, their error
    against the oracle's accurate FP64 product."""
    import oracle as O
    y = np.zeros(A.n_rows)
    O.crs_spmv_omp(A, x, y)  # first touch
    times = []
    t_all = time.perf_counter()
    while True:
        t0 = time.perf_counter()
        O.crs_spmv_omp(A, x, y)
        times.append(time.perf_counter() - t0)
        el = time.perf_counter() - t_all
        if (el >= seconds and len(times) >= 5) or len(times) >= 200:
            break
    per = statistics.median(times)
    out = {"value": round(2.0 * A.nnz / per / 1e9, 3), "unit": "GFlop/s",
           "cores": O.num_threads(), "kind": "oracle",
           "cores_in_affinity_mask": AFFINITY_CORES,
           "omp": {k: os.environ.get(k) for k in ("OMP_PROC_BIND", "OMP_PLACES")},
           "sample": f"full matrix, median of {len(times)} SpMVMs with the OpenMP static CRS loop ({el:.1f} s)"}
    t0 = time.perf_counter()
    O.crs_spmv(A, x)
    out["serial_crs_gflops"] = round(2.0 * A.nnz / (time.perf_counter() - t0) / 1e9, 3)
    J = O.jds_build(A, symmetric=True)
    xp = O.permute(J.perm, x)
    t0 = time.perf_counter()
    O.jds_spmv(J, xp)
    out["serial_jds_gflops"] = round(2.0 * A.nnz / (time.perf_counter() - t0) / 1e9, 3)
    out["serial_cores"] = 1
    out["host_copy_gbs"] = host_copy_gbs()
    if fp32_products is not None:
        out["fp32_error_vs_oracle"] = fp32_error_vs_oracle(fp32_products)
    return out


def run_reference(args):
    world, rank, _ = dist_env()
    if rank != 0:
        return None
    A, x = make_workload(args.config)
    import oracle as O
    y = np.zeros(A.n_rows)
    O.crs_spmv_omp(A, x, y)
    for _ in range(max(args.warmup, 3)):
        O.crs_spmv_omp(A, x, y)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        O.crs_spmv_omp(A, x, y)
    el = time.perf_counter() - t0
    per = el / args.steps
    val = round(2.0 * A.nnz / per / 1e9, 3)
    return {"metric": METRIC, "value": val, "unit": "GFlop/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": round(per * 1e3, 3), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "impl": "reference",
            "config": {"workload": WORKLOADS.get(args.config, WORKLOAD), "config_index": args.config, "n_rows": A.n_rows,
                       "nnz": A.nnz, "kernel": "oracle CRS loop, OpenMP static schedule"},
            "cpu_baseline": {"value": val, "unit": "GFlop/s", "cores": O.num_threads(),
                             "kind": "oracle", "sample": f"full matrix, {args.steps} timed SpMVMs"},
            "e2e": {"value": val, "unit": "GFlop/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}


def run_micro(args):
    """The basic sparse vector operations of Sect. 4.1 on the device: the
    table of ADD / SCP over packed dense (PD), constant stride (CS) and
    indirect (IS: ind(i) = k i; IR: random strides of mean k, as the paper
    draws them) access at the paper's strides 1, 8 and 530; the IS / IR
    stride sweep; and IR with Gaussian strides over a mean/variance plane.
    Each point: median of 7 launches, L2 flushed (a 512 MB write) before
    each, CUDA events around the launch only."""
    import torch
    from paper_0910_4836_gb300 import build, synth as S
    from paper_0910_4836_gb300.gather import GatherSum
    build()
    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    stream = torch.cuda.current_stream(dev)
    flush = torch.empty(64 * 2 ** 20, dtype=torch.float64, device=dev)
    i32max = 2 ** 31 - 1
    gen = torch.Generator(device=dev)
    gen.manual_seed(11)
    B = torch.rand(i32max + 1, dtype=torch.float64, device=dev, generator=gen)
    A = torch.rand(2 ** 26, dtype=torch.float64, device=dev, generator=gen)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)

    def timed(g):
        t = []
        for _ in range(7):
            flush.fill_(1.0)
            e0.record(stream)
            g()
            e1.record(stream)
            e1.synchronize()
            t.append(e0.elapsed_time(e1))
        return statistics.median(t)

    def point(op, access, n, k=1, ind=None):
        ind_d = None if ind is None else torch.as_tensor(ind).to(dev)
        g = GatherSum(op, access, n, B, a=A[:n] if op == "SCP" else None, k=k, ind=ind_d)
        ms = timed(g)
        useful = n * (8 + (8 if op == "SCP" else 0) + (4 if access in ("IND", "IND_TMA") else 0))
        res = {"n": n, "us": round(ms * 1e3, 2), "gups": round(n / (ms * 1e-3) / 1e9, 2),
               "useful_gbs": round(useful / (ms * 1e-3) / 1e9, 1)}
        return res

    def n_for(k, cap=2 ** 26):
        return int(min(cap, 0.9 * i32max / k))

    table = {}
    for op in ("ADD", "SCP"):
        table[f"PD{op}"] = point(op, "PD", 2 ** 26)
        for k in (8, 530):
            n = n_for(k)
            table[f"CS{op} k={k}"] = point(op, "CS", n, k=k)
            table[f"IS{op} k={k}"] = point(op, "IND", n, ind=S.stride_indices(n, k))
        for k in (1, 8, 530):
            n = n_for(k)
            table[f"IR{op} k={k}"] = point(op, "IND", n, ind=S.geometric_indices(n, 1.0 / k, 100 + k))
    sweep = {}
    for k in (1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 530, 1024):
        n = n_for(k, 2 ** 25)
        sweep[str(k)] = {"ISSCP": point("SCP", "IND", n, ind=S.stride_indices(n, k)),
                         "IRSCP": point("SCP", "IND", n, ind=S.geometric_indices(n, 1.0 / k, 200 + k))}
    # the x gathers of the Zipf-rows workload (22.1M entries, uniform random
    # columns over 4M rows): one load per lane (IND) against TMA gather4
    # copies into shared memory (IND_TMA), and the floor of a column-panel
    # design, in which every SM reads all of x through shared memory
    from paper_0910_4836_gb300.gather import stage_sweep
    nz, lz = 22_098_169, 4_000_000
    zind = S.uniform_indices(nz, lz, 401)
    zipf_like = {"n": nz, "vector": lz}
    for op in ("ADD", "SCP"):
        for acc in ("IND", "IND_TMA"):
            zipf_like[f"{op} {acc}"] = point(op, acc, nz, ind=zind)
    xs = B[:lz]
    ms = timed(lambda: stage_sweep(xs))
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    zipf_like["stage_sweep"] = {"us": round(ms * 1e3, 1), "sms": sms,
                                "l2_to_smem_tbs": round(sms * lz * 8 / (ms * 1e-3) / 1e12, 2),
                                "what": "every SM reads all of x through shared memory once"}
    table["zipf_like_gathers"] = zipf_like
    plane = {}
    n = 2 ** 23
    for mean in (1, 4, 16, 64, 256):
        length = min(n * mean, i32max)
        for var in (0, 1, 16, 256, 4096, 65536):
            ind = S.gaussian_indices(n, float(mean), float(var), length, 300 + mean)
            plane[f"mean={mean} var={var}"] = point("SCP", "IND", n, ind=ind)
    return {"metric": "basic gather operations (Sect. 4.1): G element updates/s", "unit": "G updates/s",
            "dtype": "f64", "data": "synthetic (torch.rand values; SplitMix64 index arrays)",
            "l2": "flushed before every launch", "table": table, "stride_sweep": sweep,
            "gaussian_plane": plane}


def run_analysis(args):
    """Sect. 4.2's analysis of the storage schemes on the bench workload: the
    stride distribution of the x accesses in storage order (Fig. 4a: CRS,
    JDS, RBJDS with block 1 and 1024, SOJDS 1024, plus SELL-32-sigma), the
    sectors per warp-wide gather of the GPU kernels, and the block-size
    sweep of NBJDS / RBJDS / SOJDS (Fig. 5) with the GPU's own knobs (CRS
    lanes x rows per warp, NUJDS unroll x rows, SELL window x unroll)."""
    import torch
    from paper_0910_4836_gb300 import CRSMatrix, build
    from paper_0910_4836_gb300.analysis import mean_sectors, stride_hist, summary, warp_sectors
    build()
    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    time_launches = _timer(dev)
    A, x_host = make_workload(args.config)
    M = CRSMatrix.from_host(A, device=dev)
    x = torch.as_tensor(x_host).to(dev)
    y = torch.empty(A.n_rows, dtype=torch.float64, device=dev)
    out = {"workload": WORKLOAD, "n_rows": A.n_rows, "nnz": A.nnz, "stride_dist": {}, "warp_sectors": {},
           "sweep": {}}

    def strides(name, col):
        f, b = stride_hist(col)
        out["stride_dist"][name] = {"forward": f.tolist(), "backward": b.tolist(), **summary(f, b)}

    def sectors(name, H, lanes=32):
        h = warp_sectors(H, lanes)
        out["warp_sectors"][name] = {"mean": round(mean_sectors(h), 3), "hist": h.tolist()}

    def basis_of(H):
        # row-only handles: the original basis (y scattered in the kernel);
        # symmetric ones: the permuted basis with x permuted; CRS: original
        return 1 if getattr(H, "symmetric", True) is False else 0

    def timed(name, H, xin, configure_fn=None):
        if configure_fn:
            configure_fn()
        b = basis_of(H)
        t = statistics.median(time_launches(lambda: H.spmv(xin, out=y, basis=b), 10))
        out["sweep"][name] = {"us": round(t * 1e3, 1), "gflops": round(2.0 * A.nnz / (t * 1e-3) / 1e9, 1)}

    # throughput against the number of CTAs in use (the GPU counterpart of
    # the paper's performance against threads per socket, Sect. 5)
    out["cta_scaling"] = {}
    alg = 12 * A.nnz + 20 * A.n_rows

    def scaling(name, H, xin, limits):
        row = {}
        b = basis_of(H)
        for lim in limits:
            H.set_grid_limit(lim)
            t = statistics.median(time_launches(lambda: H.spmv(xin, out=y, basis=b), 10))
            row[str(lim or "all")] = {"us": round(t * 1e3, 1), "gbs": round(alg / (t * 1e-3) / 1e9, 1)}
        H.set_grid_limit(0)
        out["cta_scaling"][name] = row

    G = M.to_jds("SELL", "row_only", window=128, unroll=4)
    scaling("SELL w=128 u=4 (1024-thread CTAs, at most 2 per SM)", G, x,
            (8, 16, 32, 48, 64, 76, 96, 128, 152, 228, 304, 0))
    del G
    J = M.to_jds("NUJDS", "row_only", unroll=2)
    scaling("NUJDS u=2 (256-thread CTAs)", J, x, (38, 76, 152, 304, 608, 1216, 2432, 0))
    del J
    M.set_kernel("vector", lanes=4, rows_per_warp=4)
    scaling("CRS vector l4 r4 (64-thread CTAs)", M, x, (152, 304, 608, 1216, 2432, 4864, 9728, 0))
    torch.cuda.empty_cache()

    strides("CRS", M.col)
    for l, r in ((1, 1), (2, 2), (4, 4), (8, 2), (16, 2), (32, 1)):
        if r == 1 or l in (2, 4):
            sectors(f"CRS lanes={l}", M, l)
        timed(f"CRS vector l{l} r{r}", M, x, lambda l=l, r=r: M.set_kernel("vector", lanes=l, rows_per_warp=r))
    for perm in ("symmetric", "row_only"):
        J = M.to_jds("JDS", perm)
        xp = J.permute(x) if perm == "symmetric" else x
        strides(f"JDS {perm}", J.col)
        sectors(f"JDS {perm}", J)
        for u, r in ((1, 1), (2, 1), (4, 1), (8, 1), (2, 2), (4, 2), (2, 4)):
            timed(f"NUJDS {perm} u={u} r={r}", J, xp,
                  lambda u=u, r=r: (J.set_format("NUJDS" if u > 1 else "JDS", unroll=u),
                                    J.set_kernel("vector", rows_per_warp=r)))
        for b in (64, 128, 256, 512, 1024, 2048, 4096):
            timed(f"NBJDS {perm} b={b}", J, xp, lambda b=b: (J.set_format("NBJDS", block=b),
                                                            J.set_kernel("vector", rows_per_warp=1)))
        del J
        torch.cuda.empty_cache()
        for fmt in ("RBJDS", "SOJDS"):
            for b in ((1, 1024) if perm == "symmetric" else ()):
                R = M.to_jds(fmt, perm, block=b)
                strides(f"{fmt} {perm} b={b}", R.col)
                del R
            for b in (64, 256, 1024, 4096):
                R = M.to_jds(fmt, perm, block=b)
                timed(f"{fmt} {perm} b={b}", R, xp)
                del R
            torch.cuda.empty_cache()
        for w in (32, 128, 1024, 8192):
            G = M.to_jds("SELL", perm, window=w)
            strides(f"SELL {perm} w={w}", G.col)
            sectors(f"SELL {perm} w={w}", G)
            xs = G.permute(x) if perm == "symmetric" else x
            for u in (1, 2, 4):
                timed(f"SELL {perm} w={w} u={u}", G, xs, lambda u=u, G=G: G.set_format("SELL", unroll=u))
            del G
            torch.cuda.empty_cache()
    return out


def run_ncu_case(args):
    """A few launches of one kernel for an ncu capture; prints nothing to
    time.  Config 1: a 2e6-row HH-like matrix (~350 MB, above the 129 MB
    L2), or with --ncu-full the full 6e6-row workload (for one-pass
    counters only); --kernel names a step candidate, or "dval" for the
    value gradient.  Config 2: the Zipf-rows matrix (345 MB) and the
    kernel named by --kernel among its candidates."""
    import torch
    from paper_0910_4836_gb300 import CRSMatrix, build, synth as S
    build()
    only = None if args.kernel == "auto" else args.kernel
    if only in ("gather IND", "gather IND_TMA", "stage sweep"):
        # the Zipf-rows x gathers as a basic gather sum (22.1M uniform
        # indices over a 4M vector), or the staging floor
        from paper_0910_4836_gb300.gather import GatherSum, stage_sweep
        xz = torch.as_tensor(S.vector(4_000_000, 2)).cuda()
        if only == "stage sweep":
            for _ in range(3):
                stage_sweep(xz)
        else:
            ind = torch.as_tensor(S.uniform_indices(22_098_169, 4_000_000, 401)).cuda()
            gs = GatherSum("ADD", only.split()[1], ind.numel(), xz, ind=ind)
            for _ in range(3):
                gs()
        torch.cuda.synchronize()
        print("ran", only)
        return
    if args.config == 2:
        A = S.config(2)
        M = CRSMatrix.from_host(A)
        x = torch.as_tensor(S.vector(A.n_cols, 2)).cuda()
        y = torch.empty(A.n_rows, dtype=torch.float64, device="cuda")
        for name, fn, _ in zipf_candidates(M, A, x, y):
            if only is not None and name != only:
                continue
            torch.cuda.synchronize()
            for _ in range(3):
                fn()
            torch.cuda.synchronize()
            print("ran", name, "on the Zipf rows")
        return
    A = S.config(1) if args.ncu_full else S.hh_like(2_000_000, 1)
    M = CRSMatrix.from_host(A)
    x = torch.as_tensor(S.vector(A.n_cols, 1)).cuda()
    y = torch.empty(A.n_rows, dtype=torch.float64, device="cuda")
    if only == "dval":
        g = torch.as_tensor(S.vector(A.n_rows, 7)).cuda()
        d = torch.empty(A.nnz, dtype=torch.float64, device="cuda")
        for _ in range(3):
            M.dval(g, x, out=d)
        torch.cuda.synchronize()
        print("ran dval")
        return
    for c in candidates(M, A, x, only):
        if only is not None and c.name != only:
            continue
        configure(c.H, c.how)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        for _ in range(3):
            c.run(y)
        torch.cuda.synchronize()
        print("ran", c.name)


def main():
    args = parse()
    if args.ncu_case:
        run_ncu_case(args)
        return
    if args.micro:
        print(json.dumps(run_micro(args)), flush=True)
        return
    if args.analysis:
        print(json.dumps(run_analysis(args)), flush=True)
        return
    res = run_reference(args) if args.impl == "reference" else run_ours(args)
    if res is not None:
        print(json.dumps(res), flush=True)


if __name__ == "__main__":
    main()
