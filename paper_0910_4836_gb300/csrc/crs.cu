// CRS products (Sect. 2, CRS kernel: y_i = sum over row i of val_j x[col_j]).
//
// VECTOR: a warp is cut into groups of L lanes; each group owns one row at a
// time and strides through its entries (lane l takes entries l, l+L, ...),
// so a warp-wide load covers 32/L adjacent rows' entries contiguously.  Each
// group keeps R rows in flight: the loads of all R rows are issued before
// any product is formed, which is what keeps enough bytes in flight to
// saturate HBM with short rows.  The partial sums are combined by a fixed
// butterfly of warp shuffles; when a group holds as many rows as it has
// lanes, by a reduce-scatter that leaves each lane one row's total (same
// tree, fewer FP64 additions: on GB300 each one is a full-rate-limited FP64
// instruction).  Rows far longer than the others (crs_row_cut) are cut out of
// their group's loop and summed by the whole warp afterwards.  With one lane
// a row (crs_short_rows) rows are sorted into three classes by length: one
// lane, eight lanes, the whole warp.
//
// RUNS: as VECTOR, but a group's rows are consecutive and its lanes stride
// through their entries as one run (below).
//
// SpMM: lanes over right-hand sides -- lane c of a group accumulates column
// c of the pass, so each entry (val, col) is read once per pass and X's row
// slice is read as one contiguous segment.
//
// All three run in CTAs of two warps, one CTA per two warps' worth of rows
// (row_grid below).
#include <algorithm>

#include "accum.cuh"
#include "internal.cuh"
#include "rows.cuh"

namespace gbsp {

constexpr int kThreads = 256;
// RUNS: row length beyond which a row is summed by the whole warp (a group's
// rows share one run, so a long row would hold its whole group).
constexpr int kRunsLongRow = 64;

// The group's R partial sums over its L lanes (R, L powers of two) and the
// stores: a reduce-scatter, in which each lane trades half of its sums with
// its partner as long as it holds several, then adds its partner's.  Lane gl
// ends with row i = gl / (L / R) (R < L) or rows (R / L) gl + q, after
// R - 1 or L - 1 (+ log2(L / R)) additions instead of R log2(L); on GB300
// each one is a full FP64 instruction.  The tree per row is the xor butterfly
// of group_reduce with some additions' operands swapped, which the merges do
// not notice: every row's sum is bit-identical to it.  Rows of the group are
// first + i step; those flagged in lmask are not stored.
template <int VM, int L, int R>
__device__ __forceinline__ void scatter_store(Acc<VM> (&acc)[R], int64_t first, int64_t step, unsigned lmask,
                                              int64_t n_rows, typename ValT<VM>::T *__restrict__ y, int64_t ldy,
                                              int accumulate) {
    const int gl = (threadIdx.x & 31) % L;
#pragma unroll
    for (int o = L / 2, h = R / 2; o > 0; o >>= 1, h >>= 1) {
        if (h > 0) {
            const bool up = (gl & o) != 0;
#pragma unroll
            for (int k = 0; k < h; ++k) {
                Acc<VM> send = up ? acc[k] : acc[k + h];
                Acc<VM> keep = up ? acc[k + h] : acc[k];
                keep.merge_shfl_xor(send, o);
                acc[k] = keep;
            }
        } else {
            acc[0].shfl_xor_merge(o);
        }
    }
    constexpr int Q = R > L ? R / L : 1, P = L > R ? L / R : 1;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int i = Q * (gl / P) + q;
        const int64_t r = first + i * step;
        if (gl % P == 0 && r < n_rows && !((lmask >> i) & 1u)) {
            if (accumulate) acc[q].add_value(y[r * ldy]);
            y[r * ldy] = acc[q].result();
        }
    }
}

// One VECTOR step (group rows first + i G, i < R): the loop over the entries,
// `len` the group's longest row.
template <int VM, int L, int R>
__device__ __forceinline__ void vector_sums(Acc<VM> (&acc)[R], const int (&k0)[R], const int (&k1)[R], int len,
                                            const int32_t *__restrict__ col,
                                            const typename ValT<VM>::T *__restrict__ val,
                                            const typename ValT<VM>::T *__restrict__ x, int64_t ldx) {
    typedef typename ValT<VM>::T T;
#pragma unroll
    for (int i = 0; i < R; ++i) acc[i].init();
    for (int j = (threadIdx.x & 31) % L; j < len; j += L) {
        int c[R];
        T v[R];
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int k = k0[i] + j;
            const bool ok = k < k1[i];
            // read-only path, not evict-first: a lane group touches a
            // sector in several iterations, so it must survive in L1/L2
            c[i] = ok ? __ldg(col + k) : -1;
            v[i] = ok ? __ldg(val + k) : T(0);
        }
#pragma unroll
        for (int i = 0; i < R; ++i)
            if (c[i] >= 0) acc[i].add(v[i], ld_vec(x + (int64_t)c[i] * ldx));
    }
}

// A VECTOR step whose warp holds a row longer than `cut` (crs_row_cut): such
// rows are left out of the groups' loops and summed afterwards by the whole
// warp.  Out of line, so that the common step keeps its registers and code
// (with the cut in the common step the 4 x 4 shape took 76 us instead of 65 us
// on the HH-like matrix of N = 1,201,200).  flags: the cut, negative to
// accumulate: one argument more, of its own for the cut, cost the common step
// registers too (27-point stencil, 4 x 2: 70.5 us against 68.6).
template <int VM, int L, int R>
__device__ __noinline__ void vector_step_cut(int64_t first, int64_t n_rows, const int32_t *__restrict__ row_ptr,
                                             const int32_t *__restrict__ col,
                                             const typename ValT<VM>::T *__restrict__ val,
                                             const typename ValT<VM>::T *__restrict__ x, int64_t ldx,
                                             typename ValT<VM>::T *__restrict__ y, int64_t ldy, int flags) {
    constexpr int G = 32 / L;
    const int cut = abs(flags), accumulate = flags < 0;
    int k0[R], k1[R];
    int len = 0;
    unsigned lmask = 0;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int64_t r = first + i * G;
        k0[i] = 0;
        k1[i] = 0;
        if (r < n_rows) {
            k0[i] = __ldg(row_ptr + r);
            k1[i] = __ldg(row_ptr + r + 1);
        }
        if (k1[i] - k0[i] > cut) {
            lmask |= 1u << i;
            k1[i] = k0[i];
        }
        len = max(len, k1[i] - k0[i]);
    }
    Acc<VM> acc[R];
    vector_sums<VM, L, R>(acc, k0, k1, len, col, val, x, ldx);
    scatter_store<VM, L, R>(acc, first, G, lmask, n_rows, y, ldy, accumulate);
    crs_warp_long_rows<VM>((threadIdx.x & 31) % L == 0, lmask, first, G, row_ptr, col, val, x, ldx, y, ldy, accumulate);
}

// The occupancy hint (stated for 256-thread CTAs; the kernel is launched in
// two-warp CTAs, see row_grid) holds the common step at the registers it
// needs on its own (48 for four rows a group, 40 for fewer): without it, the
// call to the long-row step raised some shapes to 60.
template <int VM, int L, int R>
__global__ void __launch_bounds__(kThreads, R == 4 ? 5 : 6)
crs_vector_kernel(int64_t n_rows, const int32_t *__restrict__ row_ptr,
                  const int32_t *__restrict__ col, const typename ValT<VM>::T *__restrict__ val,
                  const typename ValT<VM>::T *__restrict__ x, int64_t ldx,
                  typename ValT<VM>::T *__restrict__ y, int64_t ldy, int flags) {
    constexpr int G = 32 / L;
    constexpr int RW = G * R;
    const int grp = (threadIdx.x & 31) / L;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t base = warp * RW; base < n_rows; base += nwarp * RW) {
        int k0[R], k1[R];
        int len = 0;
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int64_t r = base + i * G + grp;
            k0[i] = 0;
            k1[i] = 0;
            if (r < n_rows) {
                k0[i] = __ldg(row_ptr + r);
                k1[i] = __ldg(row_ptr + r + 1);
            }
            len = max(len, k1[i] - k0[i]);
        }
        if (__reduce_max_sync(0xffffffffu, (unsigned)len) > (unsigned)abs(flags)) {
            if constexpr (L == 1)
                short_rows_cut<VM, kShortRows>(kShortRows, base, min(base + RW, n_rows), row_ptr, col, val, x, ldx, y, ldy,
                                               flags < 0);
            else
                vector_step_cut<VM, L, R>(base + grp, n_rows, row_ptr, col, val, x, ldx, y, ldy, flags);
            continue;
        }
        Acc<VM> acc[R];
        vector_sums<VM, L, R>(acc, k0, k1, len, col, val, x, ldx);
        scatter_store<VM, L, R>(acc, base + grp, G, 0u, n_rows, y, ldy, flags < 0);
    }
}

// VECTOR with one lane a row, one or two sets of 32 consecutive rows a warp
// (four: crs_vector_kernel).  With one set, rows of every class are expected
// and taken in line.  With two, a step whose rows are all short has registers
// of its own (40, 48 warps an SM), two slots of both sets at a time.  One set
// / two, FP64: Zipf rows, 4M, 170 / 196 us; the remainder of a hybrid matrix
// (6M rows, 5.0 entries a row, at most 17) 158 / 125 us; rows of U{1..5} 40 /
// 34 us; 5-point Laplacian 1000 x 1000 16.9 / 15.2 us.
template <int VM, int R, int CUT>
__global__ void __launch_bounds__(kThreads, 6)
crs_short_kernel(int cut, int64_t n_rows, const int32_t *__restrict__ row_ptr,
                 const int32_t *__restrict__ col, const typename ValT<VM>::T *__restrict__ val,
                 const typename ValT<VM>::T *__restrict__ x, int64_t ldx,
                 typename ValT<VM>::T *__restrict__ y, int64_t ldy, int accumulate) {
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t base = warp * 32 * R; base < n_rows; base += nwarp * 32 * R) {
        if (R == 1) {
            crs_short_rows<VM, CUT>(cut, base, n_rows, row_ptr, col, val, x, ldx, y, ldy, accumulate);
            continue;
        }
        const int64_t first = base + (threadIdx.x & 31);
        int k0[R], n[R], len = 0;
#pragma unroll
        for (int i = 0; i < R; ++i) {
            k0[i] = 0;
            n[i] = 0;
            if (first + 32 * i < n_rows) {
                k0[i] = __ldg(row_ptr + first + 32 * i);
                n[i] = __ldg(row_ptr + first + 32 * i + 1) - k0[i];
            }
            len = max(len, n[i]);
        }
        const int longest = (int)__reduce_max_sync(0xffffffffu, (unsigned)len);
        if (longest > (CUT > 0 ? CUT : cut)) {
            short_rows_cut<VM, CUT>(cut, base, min(base + 32 * R, n_rows), row_ptr, col, val, x, ldx, y, ldy, accumulate);
            continue;
        }
        Acc<VM> acc[R];
        lane_sums<VM, R, 2>(acc, k0, n, col, val, x, ldx, longest);
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int64_t r = first + 32 * i;
            if (r < n_rows) {
                if (accumulate) acc[i].add_value(y[r * ldy]);
                y[r * ldy] = acc[i].result();
            }
        }
    }
}

// Park a lane's running sum in its row's slot.  Indices are compile-time
// after unrolling, so the slots stay in registers (selects, no FP64 work).
template <int VM, int R>
__device__ __forceinline__ void park(Acc<VM> (&part)[R], int cur, const Acc<VM> &acc) {
#pragma unroll
    for (int m = 0; m < R; ++m)
        if (m == cur) part[m] = acc;
}

// RUNS: the R rows of a lane group are consecutive, so CRS stores their
// entries as one contiguous run, and the group's L lanes stride through that
// whole run (lane l takes run entries l, l+L, ...) instead of through each
// row up to the longest row's length.  A lane keeps one running FMA chain
// and parks it in the row's slot when its next entry lies in a later row
// (each row is one stretch of the run, so a slot is written once; register
// selects, no FP64 work); the slots are then combined over the group by the
// reduce-scatter, after which lane l holds rows (R/L) l .. (R/L) l + R/L - 1.
// FP64 lane-slots per warp: 32 x the longest group run / L, plus R (1 - 1/L)
// additions per lane, where VECTOR pays R x 32 x the longest row / L.  U
// entries per lane are loaded and gathered before any product is formed (U
// gathers in flight).
constexpr int kRunsU = 4;

// A RUNS step whose warp holds a row longer than kRunsLongRow: such rows are
// cut out of their group's run (its index skips them: run index j of row i
// sits at entry j + b_i - p_i, p_i the run length before row i) and summed
// afterwards by the whole warp.  Out of line, so that the common step keeps
// its code.
template <int VM, int L, int R>
__device__ __noinline__ void runs_step_cut(int64_t rg, int64_t n_rows, const int32_t *__restrict__ row_ptr,
                                           const int32_t *__restrict__ col,
                                           const typename ValT<VM>::T *__restrict__ val,
                                           const typename ValT<VM>::T *__restrict__ x, int64_t ldx,
                                           typename ValT<VM>::T *__restrict__ y, int64_t ldy, int accumulate) {
    typedef typename ValT<VM>::T T;
    constexpr int U = kRunsU;
    const int gl = (threadIdx.x & 31) % L;
    int b[R + 1], p[R];  // row pointers; run index of each row's start
#pragma unroll
    for (int i = 0; i <= R; ++i) b[i] = __ldg(row_ptr + min(rg + i, n_rows));
    unsigned lmask = 0;
    int n = 0;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        p[i] = n;
        const int li = b[i + 1] - b[i];
        if (li > kRunsLongRow) lmask |= 1u << i;
        else n += li;
    }
    Acc<VM> part[R];
#pragma unroll
    for (int i = 0; i < R; ++i) part[i].init();
    Acc<VM> acc;
    acc.init();
    int cur = 0;
    for (int j = gl; j < n; j += U * L) {
        int c[U], row[U];
        T v[U], xv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int jj = j + u * L;
            // the last row starting at or before jj (a cut-out or empty row
            // starts where the next one does, which then wins)
            int i = 0, k = jj + b[0];
#pragma unroll
            for (int m = 1; m < R; ++m)
                if (jj >= p[m]) {
                    i = m;
                    k = jj + b[m] - p[m];
                }
            row[u] = i;
            const bool ok = jj < n;
            c[u] = ok ? __ldg(col + k) : -1;
            v[u] = ok ? __ldg(val + k) : T(0);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) xv[u] = c[u] >= 0 ? ld_vec(x + (int64_t)c[u] * ldx) : T(0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (c[u] >= 0) {
                if (row[u] != cur) {
                    park<VM, R>(part, cur, acc);
                    acc.init();
                    cur = row[u];
                }
                acc.add(v[u], xv[u]);
            }
        }
    }
    park<VM, R>(part, cur, acc);
    scatter_store<VM, L, R>(part, rg, 1, lmask, n_rows, y, ldy, accumulate);
    crs_warp_long_rows<VM>(gl == 0, lmask, rg, 1, row_ptr, col, val, x, ldx, y, ldy, accumulate);
}

template <int VM, int L, int R>
__global__ void __launch_bounds__(kThreads, R == 4 ? 5 : 4)
crs_runs_kernel(int64_t n_rows, const int32_t *__restrict__ row_ptr,
                const int32_t *__restrict__ col, const typename ValT<VM>::T *__restrict__ val,
                const typename ValT<VM>::T *__restrict__ x, int64_t ldx,
                typename ValT<VM>::T *__restrict__ y, int64_t ldy, int accumulate) {
    typedef typename ValT<VM>::T T;
    static_assert(R >= L && R % L == 0, "a group's rows must divide over its lanes");
    constexpr int G = 32 / L;
    constexpr int RW = G * R;
    constexpr int U = kRunsU;
    const int lane = threadIdx.x & 31;
    const int grp = lane / L, gl = lane % L;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t base = warp * RW; base < n_rows; base += nwarp * RW) {
        const int64_t rg = base + (int64_t)grp * R;
        int b[R + 1];
#pragma unroll
        for (int i = 0; i <= R; ++i) b[i] = __ldg(row_ptr + min(rg + i, n_rows));
        int longest = 0;
#pragma unroll
        for (int i = 0; i < R; ++i) longest = max(longest, b[i + 1] - b[i]);
        if (__reduce_max_sync(0xffffffffu, (unsigned)longest) > (unsigned)kRunsLongRow) {
            runs_step_cut<VM, L, R>(rg, n_rows, row_ptr, col, val, x, ldx, y, ldy, accumulate);
            continue;
        }
        Acc<VM> part[R];
#pragma unroll
        for (int i = 0; i < R; ++i) part[i].init();
        Acc<VM> acc;
        acc.init();
        int cur = 0;
        const int k0 = b[0], n = b[R] - b[0];
        for (int j = gl; j < n; j += U * L) {
            int c[U];
            T v[U], xv[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool ok = j + u * L < n;
                c[u] = ok ? __ldg(col + k0 + j + u * L) : -1;
                v[u] = ok ? __ldg(val + k0 + j + u * L) : T(0);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) xv[u] = c[u] >= 0 ? ld_vec(x + (int64_t)c[u] * ldx) : T(0);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (c[u] >= 0) {
                    const int k = k0 + j + u * L;
                    int i = 0;
#pragma unroll
                    for (int m = 1; m < R; ++m) i += k >= b[m] ? 1 : 0;
                    if (i != cur) {
                        park<VM, R>(part, cur, acc);
                        acc.init();
                        cur = i;
                    }
                    acc.add(v[u], xv[u]);
                }
            }
        }
        park<VM, R>(part, cur, acc);
        scatter_store<VM, L, R>(part, rg, 1, 0u, n_rows, y, ldy, accumulate);
    }
}

constexpr int kRowCta = 64;  // see row_grid

// SpMM: the lanes of a warp form 32 / W groups of W lanes, one lane per
// right-hand side of the pass.  FP64: a warp takes up to 16 rows and the
// groups take them by length (spmm_rows): bound by FP64 issue (90% of it on
// the HH-like matrix, N = 1,201,200: k = 16 487 -> 452 us, k = 5 281 -> 182
// us, k = 3 158 -> 131 us; rows of one length only lose by it, 5% at 1.2M rows
// of 27).  Few rows a warp keep the rows that are in work at one time close
// together: 32 instead of 16 took 540 us, X's rows leaving L2 before the other
// diagonals come back to them; fewer than 64 warps an SM (more than 32
// registers) cost as much as longer steps gain.  Fewer rows still where 16
// would not fill the GPU twice (launch_spmm).  Where the groups cover those
// rows in one round, with one group a warp, which pairs nothing, and in FP32,
// which is not bound by FP64 issue, a group takes one row in matrix order.
template <int VM, int W>
__host__ __device__ constexpr int spmm_rows_per_warp() {
    return VM == VM_F64 && 32 / W > 1 && 32 / W < 16 ? 16 / (32 / W) * (32 / W) : 32 / W;
}

template <int VM, int W>
__global__ void __launch_bounds__(kThreads, spmm_rows_per_warp<VM, W>() > 32 / W ? 8 : 0)
crs_spmm_kernel(int64_t n_rows, const int32_t *__restrict__ row_ptr,
                const int32_t *__restrict__ col, const typename ValT<VM>::T *__restrict__ val,
                const typename ValT<VM>::T *__restrict__ X, int64_t ldx,
                typename ValT<VM>::T *__restrict__ Y, int64_t ldy, int k, int c0, int accumulate, int rw) {
    typedef typename ValT<VM>::T T;
    __shared__ uint8_t order[kRowCta / 32][32];
    constexpr int G = 32 / W, RW = spmm_rows_per_warp<VM, W>();
    const int lane = threadIdx.x & 31, grp = lane / W, cc = c0 + lane % W;
    const bool active = grp < G && cc < k;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (RW > G) {
        if (warp * rw < n_rows)
            spmm_rows<VM, W>(warp * rw, (int)min((int64_t)rw, n_rows - warp * rw), active, order[threadIdx.x >> 5],
                             row_ptr, col, val, X + cc, ldx, Y + cc, ldy, accumulate);
        return;
    }
    for (int64_t r = warp * G + grp; r - grp < n_rows; r += ((int64_t)gridDim.x * blockDim.x >> 5) * G) {
        if (r >= n_rows || grp >= G) continue;
        const int k0 = __ldg(row_ptr + r), k1 = __ldg(row_ptr + r + 1);
        Acc<VM> acc;
        acc.init();
        int j = k0;
        for (; j + 4 <= k1; j += 4) {
            int ci[4];
            T vi[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                ci[u] = __ldg(col + j + u);
                vi[u] = __ldg(val + j + u);
            }
            if (active) {
#pragma unroll
                for (int u = 0; u < 4; ++u) acc.add(vi[u], ld_vec(X + (int64_t)ci[u] * ldx + cc));
            }
        }
        for (; j < k1; ++j) {
            const int ci = __ldg(col + j);
            const T vi = __ldg(val + j);
            if (active) acc.add(vi, ld_vec(X + (int64_t)ci * ldx + cc));
        }
        if (active) {
            T *yp = Y + r * ldy + cc;
            if (accumulate) acc.add_value(*yp);
            *yp = acc.result();
        }
    }
}

// dval_k: d = (accumulate ? dval_k : 0), then d = fma(G[row_k, t], X[col_k, t], d)
// for t = 0, 1, ..., m-1 (m = 1: g[row] x[col]).  One running sum in a fixed
// order, so splitting the t range over several calls changes nothing.
// Both kernels give a warp 32 consecutive rows and walk their entries in
// chunks of 32: lane l takes entry c + l of chunk c, so every col load and
// dval store is one contiguous warp-wide access.
//   m = 1 (crs_dval_kernel): kDvalU chunks in flight together (their
//     gathers are what the kernel waits for); the warp's 32 row starts and
//     ends sit one per lane, and a lane finds its entry's row from one
//     warp-wide OR of the rows' start positions in the chunk and one ballot
//     (no shuffles: a five-step shuffle search per chunk took 42% of the
//     L1TEX data-pipe wavefronts); dval is written evict-first (it is not
//     read again here), which leaves L2 to the gathered vectors.
//   m > 1 (crs_dval_multi_kernel): one chunk at a time, rows found by
//     stepping forward through the row pointers in shared memory; for m
//     = 2 .. 6 the steps' loads are issued together.  27-point stencil
//     against the loop over m: m = 2 176 -> 128 us, m = 5 247 -> 239, m = 6 346 ->
//     285 (FP64 issue alone takes 86, 215 and 258); FP32 m = 5 181 -> 136.
//     From seven steps on FP64 issue hides the loop's latency (m = 7 and 8 as
//     instances 2% faster; FP32 would gain there still: 400,000 rows of 27,
//     m = 7, 80 against 54 us); four steps at a time gained nothing (m = 8 387
//     against 375 us).  Registers for four CTAs an SM: without the hint the
//     loads do not all stay in flight (Zipf rows, 1M, m = 5 and 6: 228 and 256
//     us, 250 and 297 without; six CTAs are no faster, but for m = 2 with
//     accumulation in FP64: 400,000 rows of 27, 64 against 76 us).  With the loop,
//     several chunks in flight took 72 registers and ran slower (m = 5: 287 us
//     against 249 us); so did the shuffle-free row lookup with one or two
//     chunks in flight (294-490 us).
constexpr int kDvalWarps = kThreads / 32;
constexpr int kDvalU = 4;

template <typename T>
__global__ void __launch_bounds__(kThreads)
crs_dval_kernel(int64_t n_rows, const int32_t *__restrict__ row_ptr,
                const int32_t *__restrict__ col, const T *__restrict__ G, int64_t g_row,
                const T *__restrict__ X, int64_t x_row, T *__restrict__ dval, int accumulate) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r0 = warp * 32; r0 < n_rows; r0 += nwarp * 32) {
        // lane i: start of row r0 + i (rows past the end start at nnz)
        const int32_t rpl = __ldg(row_ptr + min(r0 + lane, n_rows));
        const int32_t e1 = __ldg(row_ptr + min(r0 + 32, n_rows));
        const int32_t eb = __shfl_sync(0xffffffffu, rpl, 0);
        const T *Gw = G + r0 * g_row;
        // lane i: end of row r0 + i
        const int32_t rpn = __ldg(row_ptr + min(r0 + lane + 1, n_rows));
        for (int32_t c = eb; c < e1; c += 32 * kDvalU) {
            int32_t cj[kDvalU], rl[kDvalU];
            T d[kDvalU];
#pragma unroll
            for (int u = 0; u < kDvalU; ++u) {
                const int32_t cb = c + 32 * u;
                const int32_t e = cb + lane;
                rl[u] = chunk_row(rpl, rpn, cb, lane);
                cj[u] = e < e1 ? ld_stream(col + e) : -1;
            }
#pragma unroll
            for (int u = 0; u < kDvalU; ++u) {
                const int32_t e = c + 32 * u + lane;
                d[u] = cj[u] >= 0 ? fma(__ldg(Gw + rl[u] * g_row), __ldg(X + (int64_t)cj[u] * x_row),
                                        accumulate ? dval[e] : T(0))
                                  : T(0);
            }
#pragma unroll
            for (int u = 0; u < kDvalU; ++u)
                if (cj[u] >= 0) __stcs(dval + c + 32 * u + lane, d[u]);
        }
    }
}

template <typename T, int M>
__global__ void __launch_bounds__(kThreads, M == 0 ? 0 : M == 2 ? 6 : 4)
crs_dval_multi_kernel(int64_t n_rows, const int32_t *__restrict__ row_ptr,
                const int32_t *__restrict__ col, int m, const T *__restrict__ G, int64_t g_row,
                int64_t g_t, const T *__restrict__ X, int64_t x_row, int64_t x_t, T *__restrict__ dval,
                int accumulate) {
    __shared__ int32_t srp[kDvalWarps][33];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t *rp = srp[wid];
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r0 = warp * 32; r0 < n_rows; r0 += nwarp * 32) {
        __syncwarp();  // the previous range's row pointers are no longer read
        rp[lane] = __ldg(row_ptr + min(r0 + lane, n_rows));
        if (lane == 0) rp[32] = __ldg(row_ptr + min(r0 + 32, n_rows));
        __syncwarp();
        const int32_t e1 = rp[32];
        int r = 0;  // local row of this lane's current entry
        for (int32_t e = rp[0] + lane; e < e1; e += 32) {
            while (rp[r + 1] <= e) ++r;  // stops at r <= 31, since e < rp[32]
            const int64_t row = r0 + r;
            const int64_t cj = ld_stream(col + e);
            T d = accumulate ? dval[e] : T(0);
            const T *gp = G + row * g_row, *xp = X + cj * x_row;
            if (M > 0) {
                T gv[M > 0 ? M : 1], xv[M > 0 ? M : 1];
#pragma unroll
                for (int t = 0; t < M; ++t) {
                    gv[t] = __ldg(gp + t * g_t);
                    xv[t] = __ldg(xp + t * x_t);
                }
#pragma unroll
                for (int t = 0; t < M; ++t) d = fma(gv[t], xv[t], d);
            } else {
                for (int t = 0; t < m; ++t) d = fma(__ldg(gp + t * g_t), __ldg(xp + t * x_t), d);
            }
            dval[e] = d;
        }
    }
}

__global__ void crs_validate_kernel(int64_t n_rows, int64_t n_cols, int64_t nnz,
                                    const int32_t *__restrict__ row_ptr,
                                    const int32_t *__restrict__ col, int32_t *status) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool bad = false;
    if (tid == 0 && (row_ptr[0] != 0 || (int64_t)row_ptr[n_rows] != nnz)) bad = true;
    for (int64_t i = tid; i < n_rows; i += stride)
        if (row_ptr[i + 1] < row_ptr[i]) bad = true;
    for (int64_t k = tid; k < nnz; k += stride) {
        const int32_t c = col[k];
        if (c < 0 || (int64_t)c >= n_cols) bad = true;
    }
    if (bad) *status = (int32_t)GBSP_ERR_MATRIX;
}

// ------------------------------------------------------------------ host --

static int grid_for(int64_t warps_needed) {
    const int64_t blocks = ceil_div(warps_needed, kThreads / 32);
    const int64_t cap = (int64_t)num_sms() * 8 * 4;  // four waves of full occupancy
    return (int)std::max<int64_t>(1, std::min(blocks, cap));
}

// The row kernels (VECTOR, RUNS, SpMM) run in CTAs of two warps, one CTA per
// two warps' worth of rows: a CTA's slot frees as soon as its two warps are
// done, instead of when the slowest of eight is, so the block scheduler
// keeps the SMs full of warps with work left.  HH-like 6M, CRS vector 4 x 4:
// 289 us against 305 us with 256-thread CTAs on a four-wave grid; Zipf
// rows 515 against 584 us; SpMM k = 16 2489 against 2680 us.
static int row_grid(int64_t warps_needed) {
    return (int)std::max<int64_t>(1, ceil_div(warps_needed, kRowCta / 32));
}

template <int VM, int L, int R>
static void launch_vector_R(const Mat &A, const VecArgs &v, cudaStream_t s) {
    typedef typename ValT<VM>::T T;
    const int grid = (int)limit_grid(row_grid(ceil_div(A.n_rows, (32 / L) * R)), A.grid_limit);
    crs_vector_kernel<VM, L, R><<<grid, kRowCta, 0, s>>>(A.n_rows, A.row_ptr, A.col, static_cast<const T *>(A.val),
                                                         static_cast<const T *>(v.x), v.ldx, static_cast<T *>(v.y),
                                                         v.ldy, v.accumulate ? -crs_row_cut(A) : crs_row_cut(A));
}

template <int VM, int L>
static void launch_vector_L(const Mat &A, const VecArgs &v, int R, cudaStream_t s) {
    if (R == 1) launch_vector_R<VM, L, 1>(A, v, s);
    else if (R == 2) launch_vector_R<VM, L, 2>(A, v, s);
    else launch_vector_R<VM, L, 4>(A, v, s);
}

template <int VM, int R, int CUT>
static void launch_short(const Mat &A, const VecArgs &v, cudaStream_t s) {
    typedef typename ValT<VM>::T T;
    const int grid = (int)limit_grid(row_grid(ceil_div(A.n_rows, 32 * R)), A.grid_limit);
    crs_short_kernel<VM, R, CUT><<<grid, kRowCta, 0, s>>>(crs_row_cut(A), A.n_rows, A.row_ptr, A.col,
                                                     static_cast<const T *>(A.val), static_cast<const T *>(v.x),
                                                     v.ldx, static_cast<T *>(v.y), v.ldy, v.accumulate);
}

template <int VM>
static void launch_vector(const Mat &A, const VecArgs &v, cudaStream_t s) {
    const int R = A.kopt.rows_per_warp;
    switch (A.kopt.lanes) {
        case 1:
            // a cut of its own (lanes = 1 asked for on longer rows): two sets
            if (crs_row_cut(A) > kShortRows) launch_short<VM, 2, 0>(A, v, s);
            else if (R == 1) launch_short<VM, 1, kShortRow>(A, v, s);
            else if (R == 2) launch_short<VM, 2, kShortRows>(A, v, s);
            else launch_vector_R<VM, 1, 4>(A, v, s);
            break;
        case 2: launch_vector_L<VM, 2>(A, v, R, s); break;
        case 4: launch_vector_L<VM, 4>(A, v, R, s); break;
        case 8: launch_vector_L<VM, 8>(A, v, R, s); break;
        case 16: launch_vector_L<VM, 16>(A, v, R, s); break;
        default: launch_vector_L<VM, 32>(A, v, R, s); break;
    }
}

template <int VM, int L, int R>
static void launch_runs_LR(const Mat &A, const VecArgs &v, cudaStream_t s) {
    typedef typename ValT<VM>::T T;
    const int grid = (int)limit_grid(row_grid(ceil_div(A.n_rows, (32 / L) * R)), A.grid_limit);
    crs_runs_kernel<VM, L, R><<<grid, kRowCta, 0, s>>>(A.n_rows, A.row_ptr, A.col, static_cast<const T *>(A.val),
                                                        static_cast<const T *>(v.x), v.ldx,
                                                        static_cast<T *>(v.y), v.ldy, v.accumulate);
}

// (lanes, rows) pairs of RUNS; gbsp_set_kernel admits exactly these.
template <int VM>
static void launch_runs(const Mat &A, const VecArgs &v, cudaStream_t s) {
    const int L = A.kopt.lanes, R = A.kopt.rows_per_warp;
    if (L == 1 && R == 4) launch_runs_LR<VM, 1, 4>(A, v, s);
    else if (L == 1) launch_runs_LR<VM, 1, 8>(A, v, s);
    else if (L == 2 && R == 4) launch_runs_LR<VM, 2, 4>(A, v, s);
    else if (L == 2) launch_runs_LR<VM, 2, 8>(A, v, s);
    else if (L == 4 && R == 4) launch_runs_LR<VM, 4, 4>(A, v, s);
    else if (L == 4) launch_runs_LR<VM, 4, 8>(A, v, s);
    else launch_runs_LR<VM, 8, 8>(A, v, s);
}

template <int VM>
static void launch_spmm(const Mat &A, const VecArgs &v, cudaStream_t s) {
    typedef typename ValT<VM>::T T;
    const int w = spmm_width(v.k, A.kopt.rhs_tile);
    with_spmm_width(w, [&](auto W) {
        constexpr int G = 32 / W.value, RW = spmm_rows_per_warp<VM, W.value>();
        // At least two waves of 64 warps an SM (16 rows a warp everywhere, us,
        // k = 16: 10,000 rows of U{1..33} 32 -> 13.5, 40,000 of 27 40 -> 36;
        // one or four waves: 150,000 rows of U{1..33} 97 or 102 against 94);
        // fewer with more groups, which take fewer rounds and of whose rows
        // more are paired (k = 4, 230,000 rows of U{1..33}: 56 with two waves, 48.5)
        const int64_t quarters = G <= 3 ? 8 : G == 4 ? 2 : 1;
        const int64_t fill = 4 * A.n_rows / ((int64_t)num_sms() * 64 * quarters);
        const int rw = (int)std::max<int64_t>(G, std::min<int64_t>(RW, fill) / G * G);
        const int grid = row_grid(ceil_div(A.n_rows, (int64_t)rw));
        for (int c0 = 0; c0 < v.k; c0 += W.value)
            crs_spmm_kernel<VM, W.value><<<grid, kRowCta, 0, s>>>(
                A.n_rows, A.row_ptr, A.col, static_cast<const T *>(A.val), static_cast<const T *>(v.x), v.ldx,
                static_cast<T *>(v.y), v.ldy, v.k, c0, v.accumulate, rw);
    });
}

// Default VECTOR shape, from the mean row length.  Few lanes a row win: on
// GB300 every addition of a lane group's reduction is a full FP64
// instruction, idle lanes issue their FMAs anyway, and in FP32 a wide group
// gathers fewer rows' neighbouring x at a time.  Measured (us, L x 4 unless
// stated; old rule -> this one):
//   mean   matrix                  FP64                    FP32 compensated
//   5.5    Zipf rows, 4M           1 lane 1098 -> 168      8 lanes 289 -> 136
//   13     HH-like, 1.2M           4 lanes 65              16 x 2 102 -> 4: 51
//   17.5   uniform random, 0.5M    4 lanes 55              32 x 2 72 -> 4: 45
//   26     27-point stencil, 1M    8 lanes 111 -> 4 x 2: 69  32 x 2 160 -> 8: 57
//   26     uniform random, 0.4M    4 lanes 61 -> 4 x 2: 58 4 lanes 53 -> 8: 45
//   50     uniform random, 0.2M    16 x 2 61 -> 8: 55      32 x 2 47 -> 8: 47
//   100    uniform random, 0.1M    32 x 2 57 -> 16: 51     32 x 2 39 -> 16: 37
// Two lines inside the 4-lane range, 4 x 4 on their other side:
//   FP64 from 24 entries a row, two rows a group: a group's rows then end
//   too far apart for four to pay.  4 x 4 / 4 x 2: HH-like, 13: 62 / 75;
//   random, 18.5: 47.3 / 47.2, 21.5: 49.4 / 49.6, 32: 55.7 / 53.5; stencil,
//   60^3: 20.7 / 16.8, 100^3: 72.3 / 68.8 (8 x 4: 77.8, though 49 at 32).
//   FP32 from 20, eight lanes: the compensated chains halve.  4 x 4 / 8 x 4:
//   HH-like, 13: 47.7 / 51.4; random, 18.5: 41.2 / 37.0, 21.5: 43.7 / 38.3,
//   32: 49.5 / 43.1; stencil 59.4 / 57.4 (plain sums 61.7 / 55.0).
// FP32 on long rows, columns at random, is bound by the loads a row has in
// flight (8M entries, 8 / 16 / 32 lanes; banded in brackets): uniform 1..127:
// 41 / 35 / 33 (23.6 / 23.1 / 23.9), log-normal of mean 60: 45 / 41 / 38 (33 /
// 32 / 32), rows of 100: 37 / 32 / 29 (17.0 / 16.7 / 18.9), of 150: 27 / 31 /
// 23.5 (23.6 / 16.9 / 16.1): 16 lanes from 55 and 32 from 120.
static double row_mean(const Mat &A) { return A.n_rows > 0 ? (double)A.nnz / (double)A.n_rows : 0.0; }

int crs_row_cut(const Mat &A) {
    const double mean = row_mean(A);
    const int L = A.kopt.lanes;
    double cut = 16.0 * L;
    if (L == 1) cut = mean >= 7 && mean <= 16 ? 2 * mean : A.kopt.rows_per_warp == 1 ? kShortRow : kShortRows;
    else if (L < 32) cut = std::max(cut, (L <= 4 ? 3 : 2) * mean);
    return (int)std::min(cut, 1e9);
}

// One lane a row: four sets of rows a warp for the shortest rows, which are
// bound by the loads in flight (one, two and four sets, us: 8M rows of one
// entry, FP64 89, 58 and 44, FP32 93, 48 and 35; 4M rows of two, FP64 50, 33
// and 33, FP32 50, 28 and 25), two for light tails in FP64 (crs_short_kernel),
// one from five entries on, where heavy tails are as likely, and in FP32, which
// pays more for the step out of line (rows of mean 2.5 with a log-normal
// tail: 43 us with one set, 55 with two).  One, too, where the rows would not
// fill the GPU with several (5-point Laplacian, 10,000, 40,000 and 160,000 rows,
// one / two sets: 2.35 / 2.87, 2.78 / 3.24, 4.40 / 4.16 us).
int crs_default_rows(const Mat &A) {
    const double mean = row_mean(A);
    if (A.kopt.lanes > 1) return 4;
    if (mean == 0 || A.n_rows < 100000) return 1;
    if (A.dtype == GBSP_F64) return mean < 1.5 ? 4 : mean < 5 ? 2 : 1;
    return mean < 2.25 ? 4 : 1;
}

void crs_default_opts(Mat &A) {
    const double mean = row_mean(A);
    const bool f64 = A.dtype == GBSP_F64;
    const int lanes = mean < 6 ? 1 : mean < 12 ? 2 : mean < (f64 ? 36 : 20) ? 4 : mean < (f64 ? 64 : 55) ? 8
                      : mean < (f64 ? 192 : 120) ? 16 : 32;
    A.kopt.kernel = GBSP_KERNEL_VECTOR;
    A.kopt.lanes = lanes;
    A.kopt.rows_per_warp = lanes == 4 && mean >= 24 ? 2 : crs_default_rows(A);
    A.default_rows = A.kind == KIND_CRS;
    A.kopt.tile = 2048;
    A.kopt.rhs_tile = 16;
    A.kopt.accum = A.dtype == GBSP_F32 ? GBSP_ACC_COMPENSATED : GBSP_ACC_PLAIN;
}

gbsp_status crs_tiled_launch(const Mat &A, const VecArgs &v, cudaStream_t s);

gbsp_status crs_launch(const Mat &A, const VecArgs &v, cudaStream_t s) {
    if (A.n_rows == 0) return GBSP_OK;
    const int vm = A.dtype == GBSP_F64 ? VM_F64
                   : (A.kopt.accum == GBSP_ACC_COMPENSATED ? VM_F32C : VM_F32);
    if (v.k == 1 && A.kopt.kernel == GBSP_KERNEL_TILED && A.tile_rows != nullptr)
        return crs_tiled_launch(A, v, s);
    if (v.k == 1 && A.kopt.kernel == GBSP_KERNEL_RUNS) {
        if (vm == VM_F64) launch_runs<VM_F64>(A, v, s);
        else if (vm == VM_F32) launch_runs<VM_F32>(A, v, s);
        else launch_runs<VM_F32C>(A, v, s);
    } else if (v.k == 1) {
        if (vm == VM_F64) launch_vector<VM_F64>(A, v, s);
        else if (vm == VM_F32) launch_vector<VM_F32>(A, v, s);
        else launch_vector<VM_F32C>(A, v, s);
    } else {
        if (vm == VM_F64) launch_spmm<VM_F64>(A, v, s);
        else if (vm == VM_F32) launch_spmm<VM_F32>(A, v, s);
        else launch_spmm<VM_F32C>(A, v, s);
    }
    GBSP_LAUNCH_CHECK("crs product kernel");
    return GBSP_OK;
}

gbsp_status crs_validate_launch(const Mat &A, int32_t *d_status, cudaStream_t s) {
    GBSP_CUDA(cudaMemsetAsync(d_status, 0, sizeof(int32_t), s));
    const int64_t work = std::max(A.n_rows, A.nnz);
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(work, kThreads),
                                                                 (int64_t)num_sms() * 8));
    crs_validate_kernel<<<grid, kThreads, 0, s>>>(A.n_rows, A.n_cols, A.nnz, A.row_ptr, A.col,
                                                  d_status);
    GBSP_LAUNCH_CHECK("crs_validate_kernel");
    return GBSP_OK;
}

template <typename T>
static void launch_dval(const Mat &A, int32_t m, const void *G, int64_t g_row, int64_t g_t,
                        const void *X, int64_t x_row, int64_t x_t, void *dval, int32_t accumulate,
                        cudaStream_t s) {
    const int grid = grid_for(ceil_div(A.n_rows, 32));
    if (m == 1)
        crs_dval_kernel<T><<<grid, kThreads, 0, s>>>(A.n_rows, A.row_ptr, A.col, static_cast<const T *>(G), g_row,
                                                     static_cast<const T *>(X), x_row, static_cast<T *>(dval),
                                                     accumulate);
    else {
        auto go = [&](auto M) {
            crs_dval_multi_kernel<T, M.value><<<grid, kThreads, 0, s>>>(
                A.n_rows, A.row_ptr, A.col, m, static_cast<const T *>(G), g_row, g_t, static_cast<const T *>(X), x_row,
                x_t, static_cast<T *>(dval), accumulate);
        };
        switch (m) {
            case 2: go(Num<2>()); break;
            case 3: go(Num<3>()); break;
            case 4: go(Num<4>()); break;
            case 5: go(Num<5>()); break;
            case 6: go(Num<6>()); break;
            default: go(Num<0>()); break;
        }
    }
}

gbsp_status crs_dval_launch(const Mat &A, int32_t m, const void *G, int64_t g_row, int64_t g_t,
                            const void *X, int64_t x_row, int64_t x_t, void *dval, int32_t accumulate,
                            cudaStream_t s) {
    if (A.n_rows == 0 || A.nnz == 0) return GBSP_OK;
    if (A.dtype == GBSP_F64) launch_dval<double>(A, m, G, g_row, g_t, X, x_row, x_t, dval, accumulate, s);
    else launch_dval<float>(A, m, G, g_row, g_t, X, x_row, x_t, dval, accumulate, s);
    GBSP_LAUNCH_CHECK("crs_dval_kernel");
    return GBSP_OK;
}

}  // namespace gbsp
