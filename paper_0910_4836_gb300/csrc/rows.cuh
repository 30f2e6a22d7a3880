// Row lookup and whole-warp row sums shared by the CRS kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "accum.cuh"

namespace gbsp {

// A compile-time count passed to a generic lambda.
template <int N> struct Num { static constexpr int value = N; };

// f(Num<n>()) for n in 1 .. M in FP64: a real branch per count, where a fixed
// count of predicated slots would issue every FP64 instruction, with no lane
// active, too.  In FP32 idle slots cost little: f(Num<M>()).
template <int VM, int M, typename F>
__device__ __forceinline__ void with_slots(int n, F f) {
    if constexpr (VM == VM_F64 && M > 1) {
        if (n < M) {
            with_slots<VM, M - 1>(n, f);
            return;
        }
    }
    f(Num<M>());
}

// The row (0..31, of a warp's 32 rows) of entry cb + lane, for a warp that
// holds its rows' starts (rs) and ends (re) one per lane; every lane takes
// part.  An entry belongs to the last nonempty row starting at or before
// it.  Row i marks position max(start_i - cb, 0) of the 32-entry chunk at
// cb when it is nonempty there (the row holding entry cb marks 0; rows
// ending by cb, empty rows and rows starting past the chunk mark nothing),
// so each marked position has exactly one row.  B: the marked positions,
// from one warp-wide OR; C: the marking rows, from one ballot.  Both are in
// increasing order, so the lane's row is the k-th set bit of C, k the
// number of marks at or below its position, less one: the first marking row
// plus k when they are consecutive (no empty rows among them), else a
// popcount halving.  No shuffles: they share the L1TEX data pipe with the
// loads.  Lanes past the warp's last entry get an unspecified row.
__device__ __forceinline__ int chunk_row(int32_t rs, int32_t re, int32_t cb, int lane) {
    const int32_t ds = max(rs - cb, 0), de = max(re - cb, 0);
    const bool mark = ds < 32 && de > ds;
    const unsigned B = __reduce_or_sync(0xffffffffu, mark ? 1u << ds : 0u);
    const unsigned C = __ballot_sync(0xffffffffu, mark);
    int k = __popc(B & (0xffffffffu >> (31 - lane))) - 1;
    int r = C ? __ffs(C) - 1 : 0;  // no marks: a chunk past the warp's entries
    if (!((C >> r) & ((C >> r) + 1))) return r + k;
    unsigned m = C;
    r = 0;
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) {
        const int n = __popc(m & ((1u << w) - 1u));
        if (n <= k) {
            k -= n;
            m >>= w;
            r += w;
        }
    }
    return r;
}

// Flagged rows with the whole warp on each row in turn.  Every lane passes
// its group's mask (bit i: row first + i * step is long; only `leader`
// lanes' masks are read); lanes stride through a row U loads deep, with the
// next step's columns loaded while this step's gathers are in flight (a step
// then waits for one latency, not two), then a full-warp sum.  U changes no
// result.  Out of line, so that it does not weigh on the common path's
// registers.  Zipf rows (4M, 22.1M entries), RUNS 4 x 4: 188 us with four
// loads and no look-ahead, 164 us with six, 178 us with eight (spills).
template <int VM, int U = 6>
__device__ __noinline__ void crs_warp_long_rows(bool leader, unsigned mask, int64_t first, int64_t step,
                                                const int32_t *__restrict__ row_ptr,
                                                const int32_t *__restrict__ col,
                                                const typename ValT<VM>::T *__restrict__ val,
                                                const typename ValT<VM>::T *__restrict__ x, int64_t ldx,
                                                typename ValT<VM>::T *__restrict__ y, int64_t ldy, int accumulate) {
    typedef typename ValT<VM>::T T;
    const int lane = threadIdx.x & 31;
    unsigned todo = __ballot_sync(0xffffffffu, leader && mask != 0);
    while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        unsigned m = __shfl_sync(0xffffffffu, mask, src);
        const int64_t f = __shfl_sync(0xffffffffu, first, src);
        while (m) {
            const int64_t r = f + (int64_t)(__ffs(m) - 1) * step;
            m &= m - 1;
            const int s0 = __ldg(row_ptr + r), s1 = __ldg(row_ptr + r + 1);
            Acc<VM> a;
            a.init();
            int c[U];
#pragma unroll
            for (int u = 0; u < U; ++u) c[u] = s0 + lane + 32 * u < s1 ? __ldg(col + s0 + lane + 32 * u) : -1;
            auto entries = [&](auto N, int j) {  // N per lane from entry j + lane on
                T v[N.value], xv[N.value];
#pragma unroll
                for (int u = 0; u < N.value; ++u) {
                    v[u] = c[u] >= 0 ? __ldg(val + j + lane + 32 * u) : T(0);
                    xv[u] = c[u] >= 0 ? ld_vec(x + (int64_t)c[u] * ldx) : T(0);
                }
                if (N.value == U) {
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int64_t k = (int64_t)j + lane + 32 * (U + u);
                        c[u] = k < s1 ? __ldg(col + k) : -1;
                    }
                }
#pragma unroll
                for (int u = 0; u < N.value; ++u)
                    if (j + lane + 32 * u < s1) a.add(v[u], xv[u]);
            };
            int j = s0;
            for (; j + 32 * U <= s1; j += 32 * U) entries(Num<U>(), j);
            if (j < s1) with_slots<VM, U>((s1 - j + 31) >> 5, [&](auto N) { entries(N, j); });
            group_reduce<32, VM>(a);
            if (lane == 0) {
                if (accumulate) a.add_value(y[r * ldy]);
                y[r * ldy] = a.result();
            }
        }
    }
}

// VECTOR with one lane a row: rows of up to `cut` entries (crs_row_cut) by one
// lane; rows of up to kMidRow by eight lanes; longer ones by the whole warp.
// Without the two upper classes a warp runs to its longest row: on the Zipf
// rows (5.5 entries a row, up to 5000) 1098 us against 168 us now (181 us with
// a fixed number of slots a step, see with_slots); what is left there is FP64
// issue (idle lanes issue too) and the latency of the longest rows.  kMidRow
// 32, 64 and 128 gave 198, 185 and 183 us.  A row's arithmetic depends on its
// length alone, so the batched product, which cuts the rows elsewhere,
// returns the same bits.
constexpr int kMidRow = 128;

// The slots of R sets of 32 rows, one row a lane, to the longest: k0[i] and
// n[i] the lane's row of set i (n < 1: none).  The loads of U slots of all
// sets are issued together.
template <int VM, int R, int U>
__device__ __forceinline__ void lane_sums(Acc<VM> (&acc)[R], const int (&k0)[R], const int (&n)[R],
                                          const int32_t *__restrict__ col,
                                          const typename ValT<VM>::T *__restrict__ val,
                                          const typename ValT<VM>::T *__restrict__ x, int64_t ldx, int longest) {
    typedef typename ValT<VM>::T T;
#pragma unroll
    for (int i = 0; i < R; ++i) acc[i].init();
    for (int j = 0; j < longest; j += U)
        with_slots<VM, U>(min(longest - j, U), [&](auto N) {
            int c[R][N.value];
            T v[R][N.value];
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int u = 0; u < N.value; ++u) {
                    const bool ok = j + u < n[i];
                    c[i][u] = ok ? __ldg(col + k0[i] + j + u) : -1;
                    v[i][u] = ok ? __ldg(val + k0[i] + j + u) : T(0);
                }
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int u = 0; u < N.value; ++u)
                    if (c[i][u] >= 0) acc[i].add(v[i][u], ld_vec(x + (int64_t)c[i][u] * ldx));
        });
}

// Rows base + i, i in the bits of `todo` (the same in every lane; lane i
// passes the row's bounds s0, s1): eight lanes a row, four rows at a time.
template <int VM>
__device__ __forceinline__ void crs_mid_rows(unsigned todo, int64_t base, int s0, int s1,
                                             const int32_t *__restrict__ col,
                                             const typename ValT<VM>::T *__restrict__ val,
                                             const typename ValT<VM>::T *__restrict__ x, int64_t ldx,
                                             typename ValT<VM>::T *__restrict__ y, int64_t ldy, int accumulate) {
    typedef typename ValT<VM>::T T;
    const int lane = threadIdx.x & 31, grp = lane >> 3, gl = lane & 7;
    while (todo) {
        unsigned t = todo;
#pragma unroll
        for (int g = 0; g < 3; ++g)
            if (g < grp) t &= t - 1;
        const int src = t ? __ffs(t) - 1 : 0;
        const int k0 = __shfl_sync(0xffffffffu, s0, src);
        int k1 = __shfl_sync(0xffffffffu, s1, src);
        if (!t) k1 = k0;
        Acc<VM> a;
        a.init();
        const int longest = (int)__reduce_max_sync(0xffffffffu, (unsigned)(k1 - k0));
        for (int j0 = 0; j0 < longest; j0 += 4 * 8)
            with_slots<VM, 4>(min((longest - j0 + 7) >> 3, 4), [&](auto N) {
                const int j = k0 + j0 + gl;
                int c[N.value];
                T v[N.value];
#pragma unroll
                for (int u = 0; u < N.value; ++u) {
                    const bool ok = j + 8 * u < k1;
                    c[u] = ok ? __ldg(col + j + 8 * u) : -1;
                    v[u] = ok ? __ldg(val + j + 8 * u) : T(0);
                }
#pragma unroll
                for (int u = 0; u < N.value; ++u)
                    if (c[u] >= 0) a.add(v[u], ld_vec(x + (int64_t)c[u] * ldx));
            });
        group_reduce<8, VM>(a);
        if (gl == 0 && t) {
            const int64_t r = base + src;
            if (accumulate) a.add_value(y[r * ldy]);
            y[r * ldy] = a.result();
        }
#pragma unroll
        for (int g = 0; g < 4; ++g) todo &= todo - 1;
    }
}

// 32 consecutive rows from `base` on, class by class, the loads of eight slots
// of the short rows issued together.  CUT: the cut where it is a constant
// (kShortRow), else 0: FP32 Zipf rows, 4M, 138 us against 148 us with the
// cut in a register.
constexpr int kShortRow = 8, kShortRows = 12;  // one set of rows a warp, several
template <int VM, int CUT>
__device__ __forceinline__ void crs_short_rows(int cut, int64_t base, int64_t n_rows,
                                               const int32_t *__restrict__ row_ptr,
                                               const int32_t *__restrict__ col,
                                               const typename ValT<VM>::T *__restrict__ val,
                                               const typename ValT<VM>::T *__restrict__ x, int64_t ldx,
                                               typename ValT<VM>::T *__restrict__ y, int64_t ldy, int accumulate) {
    typedef typename ValT<VM>::T T;
    constexpr int U = 8;
    if (CUT > 0) cut = CUT;
    const int64_t r = base + (threadIdx.x & 31);
    int k0 = 0, n = 0, len = 0;
    if (r < n_rows) {
        k0 = __ldg(row_ptr + r);
        n = __ldg(row_ptr + r + 1) - k0;
    }
    if (n <= cut) len = n;
    Acc<VM> acc;
    acc.init();
    const int longest = (int)__reduce_max_sync(0xffffffffu, (unsigned)len);
    for (int j = 0; j < longest; j += U)
        with_slots<VM, U>(min(longest - j, U), [&](auto N) {
            int c[N.value];
            T v[N.value];
#pragma unroll
            for (int u = 0; u < N.value; ++u) {
                const bool ok = j + u < n && n <= cut;
                c[u] = ok ? __ldg(col + k0 + j + u) : -1;
                v[u] = ok ? __ldg(val + k0 + j + u) : T(0);
            }
#pragma unroll
            for (int u = 0; u < N.value; ++u)
                if (c[u] >= 0) acc.add(v[u], ld_vec(x + (int64_t)c[u] * ldx));
        });
    if (r < n_rows && n <= cut) {
        if (accumulate) acc.add_value(y[r * ldy]);
        y[r * ldy] = acc.result();
    }
    const unsigned mid = __ballot_sync(0xffffffffu, n > cut && n <= kMidRow);
    if (mid) crs_mid_rows<VM>(mid, base, k0, k0 + n, col, val, x, ldx, y, ldy, accumulate);
    const unsigned big = __ballot_sync(0xffffffffu, n > cut && n > kMidRow);
    if (big)
        crs_warp_long_rows<VM, 4>((threadIdx.x & 31) == 0, big, base, 1, row_ptr, col, val, x, ldx, y, ldy, accumulate);
}

// The 32-row sets of [base, end), out of line.
template <int VM, int CUT>
__device__ __noinline__ void short_rows_cut(int cut, int64_t base, int64_t end, const int32_t *__restrict__ row_ptr,
                                            const int32_t *__restrict__ col,
                                            const typename ValT<VM>::T *__restrict__ val,
                                            const typename ValT<VM>::T *__restrict__ x, int64_t ldx,
                                            typename ValT<VM>::T *__restrict__ y, int64_t ldy, int accumulate) {
    for (; base < end; base += 32)
        crs_short_rows<VM, CUT>(cut, base, end, row_ptr, col, val, x, ldx, y, ldy, accumulate);
}

// SpMM: lanes per row of a pass over k right-hand sides, at most `tile` (16
// when unset) of them a pass, in passes of equal width: the widest groups
// that leave as many groups to a warp (32 / width) as the pass's columns do.
__host__ __device__ inline int spmm_width(int k, int tile) {
    const int t = tile > 0 ? (tile < 32 ? tile : 32) : 16;
    const int passes = (k + t - 1) / t;
    return 32 / (32 / ((k + passes - 1) / passes));
}

// Calls f(Num<W>()) for the width w >= 2 of spmm_width.
template <typename F>
__host__ __device__ __forceinline__ void with_spmm_width(int w, F f) {
    if (w <= 2) f(Num<2>());
    else if (w <= 3) f(Num<3>());
    else if (w <= 4) f(Num<4>());
    else if (w <= 5) f(Num<5>());
    else if (w <= 6) f(Num<6>());
    else if (w <= 8) f(Num<8>());
    else if (w <= 10) f(Num<10>());
    else if (w <= 16) f(Num<16>());
    else f(Num<32>());
}

// SpMM: rows [r0, r0 + nr), nr <= 32, of one warp, whose lanes form 32 / W
// groups of W lanes, one lane per right-hand side of the pass (X and Y point
// at its column; idle lanes pass active = false).  The groups take one row
// each per round, rows in order of decreasing length, so that the rows of a
// round are about equally long: in matrix order the groups of a warp wait
// for its longest row, and an FP64 instruction costs the same however many of
// its lanes are active, even none.  Hence also the exact tail in FP64: with
// four predicated slots a step the HH-like matrix took 8.7M warp-wide FMAs for
// k = 16, with the tail 7.8M (7.6M is one full warp each).  Every row is one
// FMA chain in entry order, whatever its round.  `order`: 32 bytes of shared
// memory of the warp.
template <int VM, int W>
__device__ __forceinline__ void spmm_rows(int64_t r0, int nr, bool active, uint8_t *order,
                                          const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                                          const typename ValT<VM>::T *__restrict__ val,
                                          const typename ValT<VM>::T *__restrict__ X, int64_t ldx,
                                          typename ValT<VM>::T *__restrict__ Y, int64_t ldy, int accumulate) {
    typedef typename ValT<VM>::T T;
    constexpr int G = 32 / W;
    const int lane = threadIdx.x & 31, grp = lane / W;
    // lane i: start and length of row r0 + i
    const int s = __ldg(row_ptr + r0 + min(lane, nr));
    const int n = lane < nr ? __ldg(row_ptr + r0 + lane + 1) - s : -1;
    int rank = 0;
    for (int i = 0; i < nr; ++i) {
        const int m = __shfl_sync(0xffffffffu, n, i);
        rank += m > n || (m == n && i < lane);
    }
    __syncwarp();
    if (lane < nr) order[rank] = (uint8_t)lane;
    __syncwarp();
    for (int t = 0; t < nr; t += G) {
        const int longest = __shfl_sync(0xffffffffu, n, order[t]);
        const bool mine = active && t + grp < nr;
        const int src = t + grp < nr ? order[t + grp] : 0;
        const int k0 = __shfl_sync(0xffffffffu, s, src);
        const int len = __shfl_sync(0xffffffffu, n, src);
        Acc<VM> acc;
        acc.init();
        const int32_t *cp = col + k0;
        const T *vp = val + k0;
        // N entries of the row from j on
        auto entries = [&](auto N, int j) {
            int c[N.value];
            T v[N.value];
#pragma unroll
            for (int u = 0; u < N.value; ++u) {
                const bool ok = mine && j + u < len;
                c[u] = ok ? __ldg(cp + j + u) : -1;
                v[u] = ok ? __ldg(vp + j + u) : T(0);
            }
#pragma unroll
            for (int u = 0; u < N.value; ++u)
                if (c[u] >= 0) acc.add(v[u], ld_vec(X + (int64_t)c[u] * ldx));
        };
        int j = 0;
        for (; j + (VM == VM_F64 ? 4 : 1) <= longest; j += 4) entries(Num<4>(), j);
        switch (VM == VM_F64 ? longest - j : 0) {
            case 3: entries(Num<3>(), j); break;
            case 2: entries(Num<2>(), j); break;
            case 1: entries(Num<1>(), j); break;
        }
        if (mine) {
            T *y = Y + (r0 + src) * ldy;
            if (accumulate) acc.add_value(*y);
            *y = acc.result();
        }
    }
}

}  // namespace gbsp
