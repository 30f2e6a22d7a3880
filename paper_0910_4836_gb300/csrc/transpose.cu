// Transposed CRS structure by a two-level column split.
//
// A^T's rows are A's columns, and inside each the entries keep A's entry
// order, so the build is a stable sort of the entries by column:
//   1. split: entries go to buckets of `width` consecutive columns, as
//      16-byte records {row, entry, column inside the bucket; value}.  A CTA
//      takes one tile; each of its warps counts and then places its own
//      contiguous part, so a warp's private counters give stable ranks
//      (warp matches in chunk and lane order) without a barrier per chunk.
//   2. bucket: one CTA per bucket counts its columns (the row pointers of
//      A^T fall out), orders the bucket in shared memory, and writes t_val,
//      t_col and tmap in their final order.
// Every array is a bit-exact function of the input.
//
// Both levels are bound by L1-to-L2 packets: a scattered store or load is
// one 32-byte packet a lane.  Hence one record store an entry in level 1,
// and in level 2 one record gather an entry and stores in output order (the
// other way round, three scattered stores an entry, took twice as long).
// Carrying row and value through level 1 costs less than gathering them by
// entry at the end (a 32-byte sector each).  HH-like N = 1,201,200 (15.7M
// entries): split 171 us, bucket 172 us, the whole build 0.45 ms against
// 1.0 ms for the byte-wise radix sort (three passes of 127 us and 247 us of
// gathers by entry), which remains for matrices past the split's limits.
#include <algorithm>

#include "internal.cuh"
#include "rows.cuh"

namespace gbsp {

constexpr int kSplitWarps = 16;
constexpr int kSplitThreads = 32 * kSplitWarps;
constexpr int kMaxBuckets = 2048;
constexpr int kMaxWidth = 8192;    // columns per bucket
constexpr int kSplitSegMax = 4064; // entries per warp of a tile: 16 x 4064 < 2^16 (16-bit counters)
constexpr int kRound = 12288;      // entries of a bucket ordered in shared memory at a time
constexpr int kShortColumn = 48;   // longest column of a round that one thread sorts
constexpr int kRankColumn = 128;   // ... that a warp ranks

// Bucket of a column (n_cols <= 2048 x 8192 = 2^24): exact for
// magic = ceil(2^40 / width).
__device__ __forceinline__ int bucket_of(int32_t c, uint64_t magic) { return (int)(((uint64_t)(uint32_t)c * magic) >> 40); }

// A record's key: row, entry and column inside the bucket, in 64 bits.
struct KeyBits {
    int c, e;  // bits of the column, of the entry
};

// The row of entry e (0 <= e < nnz): the last one that starts at or before it,
// by all lanes of a warp, 32 probes a step.
__device__ __forceinline__ int64_t row_at(int64_t n_rows, const int32_t *__restrict__ row_ptr, int64_t e) {
    int64_t lo = 0, hi = n_rows;  // row_ptr[lo] <= e < row_ptr[hi]
    while (hi - lo > 1) {
        const int64_t step = (hi - lo + 31) / 32, p = lo + step * ((threadIdx.x & 31) + 1);
        lo += step * __popc(__ballot_sync(0xffffffffu, p < hi && __ldg(row_ptr + min(p, n_rows)) <= e));
        hi = min(hi, lo + step);
    }
    return lo;
}

// Row of every entry, a warp per 32 rows, 32 consecutive entries per store.
__global__ void __launch_bounds__(256)
row_of_kernel(int64_t n_rows, const int32_t *__restrict__ row_ptr, int32_t *__restrict__ row_of) {
    const int lane = threadIdx.x & 31;
    const int64_t r0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32;
    if (r0 >= n_rows) return;
    const int32_t rs = __ldg(row_ptr + min(r0 + lane, n_rows));
    const int32_t re = __ldg(row_ptr + min(r0 + lane + 1, n_rows));
    const int32_t eb = __shfl_sync(0xffffffffu, rs, 0), e1 = __shfl_sync(0xffffffffu, re, 31);
    for (int32_t c = eb; c < e1; c += 32) {
        const int r = chunk_row(rs, re, c, lane);
        if (c + lane < e1) row_of[c + lane] = (int32_t)(r0 + r);
    }
}

// The same, a CTA per kRowTile entries, whatever the rows' lengths: the tile's
// rows mark their first entries and a maximum scan spreads the marks.  For
// long rows (row_of_launch), whose warps above are few.
constexpr int kRowTile = 2048;
__global__ void __launch_bounds__(256)
row_of_tile_kernel(int64_t n_rows, int64_t nnz, const int32_t *__restrict__ row_ptr, int32_t *__restrict__ row_of) {
    __shared__ int32_t mark[kRowTile], sums[8];
    __shared__ int64_t ends[2];
    constexpr int P = kRowTile / 256;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int64_t e0 = (int64_t)blockIdx.x * kRowTile;
    const int n = (int)min((int64_t)kRowTile, nnz - e0);
    if (wid < 2) {
        const int64_t r = row_at(n_rows, row_ptr, wid == 0 ? e0 : e0 + n - 1);
        if (lane == 0) ends[wid] = r;
    }
#pragma unroll
    for (int u = 0; u < P; ++u) mark[tid + 256 * u] = 0;
    __syncthreads();
    const int64_t r0 = ends[0], r1 = ends[1];
    // of the rows that start at one entry the last has it, the others are empty
    for (int64_t r = r0 + 1 + tid; r <= r1; r += 256)
        atomicMax(mark + (__ldg(row_ptr + r) - (int32_t)e0), (int32_t)(r - r0));
    __syncthreads();
    int32_t m[P];
#pragma unroll
    for (int u = 0; u < P; ++u) {
        m[u] = mark[tid * P + u];
        if (u > 0) m[u] = max(m[u], m[u - 1]);
    }
    int32_t incl = m[P - 1];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) incl = max(incl, __shfl_up_sync(0xffffffffu, incl, o));
    if (lane == 31) sums[wid] = incl;
    int32_t before = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) before = 0;
    __syncthreads();
    for (int w = 0; w < wid; ++w) before = max(before, sums[w]);
#pragma unroll
    for (int u = 0; u < P; ++u) mark[tid * P + u] = max(before, m[u]);
    __syncthreads();
    for (int i = tid; i < n; i += 256) row_of[e0 + i] = (int32_t)r0 + mark[i];
}

// The whole transpose, rows / tiles: 30 rows of 100,000 entries 5.85 / 0.17
// ms, 300 of 3000 0.30 / 0.10, 300,000 of 100 3.32 / 3.35, 1.2M of 13 0.42 /
// 0.45.
void row_of_launch(const Mat &A, int32_t *row_of, cudaStream_t s) {
    if (A.nnz >= 128 * A.n_rows)
        row_of_tile_kernel<<<(unsigned)ceil_div(A.nnz, kRowTile), 256, 0, s>>>(A.n_rows, A.nnz, A.row_ptr, row_of);
    else
        row_of_kernel<<<(unsigned)ceil_div(A.n_rows, 256), 256, 0, s>>>(A.n_rows, A.row_ptr, row_of);
}

// Entries per (bucket, tile): counts[bucket * tiles + tile].
__global__ void __launch_bounds__(kSplitThreads)
split_count_kernel(int64_t nnz, uint64_t magic, int buckets, int64_t tiles, int64_t tile, const int32_t *__restrict__ col,
                   int32_t *__restrict__ counts) {
    __shared__ int32_t cnt[kMaxBuckets];
    for (int b = threadIdx.x; b < buckets; b += kSplitThreads) cnt[b] = 0;
    __syncthreads();
    const int64_t lo = (int64_t)blockIdx.x * tile, hi = min(lo + tile, nnz);
    for (int64_t e = lo + threadIdx.x; e < hi; e += 4 * kSplitThreads) {
        int32_t c[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) c[u] = e + u * kSplitThreads < hi ? __ldg(col + e + u * kSplitThreads) : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (c[u] >= 0) atomicAdd(&cnt[bucket_of(c[u], magic)], 1);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < buckets; b += kSplitThreads) counts[(int64_t)b * tiles + blockIdx.x] = cnt[b];
}

// Counters of one warp: 16 bits a key, two keys to a word.
__device__ __forceinline__ void count_key(uint32_t *cnt, int key, unsigned n) {
    atomicAdd(cnt + (key >> 1), n << (16 * (key & 1)));
}
__device__ __forceinline__ int read_key(const uint32_t *cnt, int key) {
    return (int)(reinterpret_cast<const volatile uint16_t *>(cnt)[key]);
}

// Stable rank of each lane's key among the keys this warp has placed, on
// top of the warp's counter, which moves past the chunk.  All lanes take
// part; idle lanes pass key < 0.
__device__ __forceinline__ int place_key(uint32_t *cnt, int key, unsigned lt) {
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    const int rank = __popc(peers & lt);
    const int at = key >= 0 ? read_key(cnt, key) + rank : 0;
    __syncwarp();
    if (key >= 0 && rank == 0) count_key(cnt, key, __popc(peers));
    __syncwarp();
    return at;
}

__device__ __forceinline__ int4 make_rec(uint64_t key, double v) {
    return make_int4((int)(uint32_t)key, (int)(uint32_t)(key >> 32), __double2loint(v), __double2hiint(v));
}
__device__ __forceinline__ int4 make_rec(uint64_t key, float v) {
    return make_int4((int)(uint32_t)key, (int)(uint32_t)(key >> 32), __float_as_int(v), 0);
}
__device__ __forceinline__ uint64_t rec_key(const int4 &r) {
    return (uint64_t)(uint32_t)r.y << 32 | (uint32_t)r.x;
}
__device__ __forceinline__ void rec_value(const int4 &r, double *v) { *v = __hiloint2double(r.w, r.z); }
__device__ __forceinline__ void rec_value(const int4 &r, float *v) { *v = __int_as_float(r.z); }

// Level 1: `seg` entries a warp, offsets[bucket * tiles + tile] the first
// place of the tile's entries in the bucket.
template <typename T>
__global__ void __launch_bounds__(kSplitThreads)
split_kernel(int64_t nnz, int width, uint64_t magic, KeyBits bits, int buckets, int64_t tiles, int seg,
             const int32_t *__restrict__ col, const int32_t *__restrict__ row_of, const T *__restrict__ val,
             const int32_t *__restrict__ offsets, int4 *__restrict__ rec) {
    extern __shared__ uint32_t split_smem[];
    const int words = (buckets + 1) / 2;
    uint32_t *cnt = split_smem;
    int32_t *base = reinterpret_cast<int32_t *>(split_smem + kSplitWarps * words);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    for (int p = threadIdx.x; p < kSplitWarps * words; p += kSplitThreads) cnt[p] = 0;
    for (int b = threadIdx.x; b < buckets; b += kSplitThreads) base[b] = __ldg(offsets + (int64_t)b * tiles + blockIdx.x);
    __syncthreads();
    const int64_t lo = ((int64_t)blockIdx.x * kSplitWarps + wid) * seg, hi = min(lo + seg, nnz);
    uint32_t *mine = cnt + wid * words;
    constexpr int U = 4;
    for (int64_t e = lo + lane; e < hi; e += 32 * U) {
        int32_t c[U];
#pragma unroll
        for (int u = 0; u < U; ++u) c[u] = e + 32 * u < hi ? __ldg(col + e + 32 * u) : -1;
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (c[u] >= 0) count_key(mine, bucket_of(c[u], magic), 1);
    }
    __syncthreads();
    // counts of every warp -> counts of the warps before it
    for (int p = threadIdx.x; p < words; p += kSplitThreads) {
        uint32_t run = 0;
#pragma unroll
        for (int w = 0; w < kSplitWarps; ++w) {
            const uint32_t v = cnt[w * words + p];
            cnt[w * words + p] = run;
            run += v;
        }
    }
    __syncthreads();
    for (int64_t c0 = lo; c0 < hi; c0 += 32 * U) {
        int32_t c[U], r[U];
        T v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t e = c0 + 32 * u + lane;
            c[u] = e < hi ? __ldg(col + e) : -1;
            r[u] = e < hi ? __ldcs(row_of + e) : 0;
            v[u] = e < hi ? __ldcs(val + e) : T(0);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int key = c[u] >= 0 ? bucket_of(c[u], magic) : -1;
            const int at = place_key(mine, key, lt);
            if (key < 0) continue;
            const uint64_t e = (uint64_t)(c0 + 32 * u + lane);
            rec[base[key] + at] =
                make_rec(((uint64_t)r[u] << bits.e | e) << bits.c | (uint32_t)(c[u] - key * width), v[u]);
        }
    }
}

// Exclusive scan of v[0..n) in place over the CTA; sums: a word a warp.
template <int THREADS>
__device__ __forceinline__ void cta_scan(int32_t *v, int n, int32_t *sums) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int per = (n + THREADS - 1) / THREADS, c0 = threadIdx.x * per, c1 = min(c0 + per, n);
    int32_t s = 0;
    for (int c = c0; c < c1; ++c) s += v[c];
    int32_t incl = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) sums[wid] = incl;
    __syncthreads();
    int32_t run = incl - s;
    for (int w = 0; w < wid; ++w) run += sums[w];
    for (int c = c0; c < c1; ++c) {
        const int32_t t = v[c];
        v[c] = run;
        run += t;
    }
    __syncthreads();
}

// The m <= kRankColumn distinct places at o in increasing order, by a warp:
// every place counts the smaller ones, a place and its rank in one register
// (the kernel has 40 for three CTAs an SM).
__device__ __forceinline__ void rank_places(uint16_t *o, int m) {
    constexpr int Q = kRankColumn / 32;
    const int lane = threadIdx.x & 31;
    uint32_t vr[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const uint32_t v = lane + 32 * q < m ? o[lane + 32 * q] : 0;
        uint32_t rank = 0;
#pragma unroll 1
        for (int i = 0; i < (32 * q < m ? m : 0); ++i) rank += o[i] < v;
        vr[q] = v << 16 | rank;
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < Q; ++q)
        if (lane + 32 * q < m) o[vr[q] & 0xffff] = (uint16_t)(vr[q] >> 16);
}

// Level 2: one CTA per bucket, in rounds of kRound records (one round unless
// columns are dense).  A round: count its columns; give every record a place
// in its column by a shared counter (in no fixed order); sort each column's
// few places back into record order, which is entry order; then write the
// round in output order.  A column with more than kShortColumn records in
// the round is sorted by a warp, one with more than kRankColumn collected in
// order by a warp in a pass over the round (all past kShortColumn: 300,000
// columns of 100 records each 3.32 ms, 2.08 ms so).
constexpr int kBucketThreads = 512;
template <typename T>
__global__ void __launch_bounds__(kBucketThreads)
bucket_kernel(int64_t n_cols, int64_t nnz, int width, KeyBits bits, int buckets, int64_t tiles,
              const int32_t *__restrict__ offsets, const int4 *__restrict__ rec, int32_t *__restrict__ t_row_ptr,
              int32_t *__restrict__ t_col, T *__restrict__ t_val, int32_t *__restrict__ tmap) {
    extern __shared__ uint32_t split_smem[];
    __shared__ int32_t sums[kBucketThreads / 32];
    __shared__ int32_t n_long;
    __shared__ int16_t longs[kRound / kShortColumn];
    int32_t *next = reinterpret_cast<int32_t *>(split_smem);  // column: place of its next record in A^T
    int32_t *start = next + width;                            // column: start in the round, moves to its end
    uint16_t *lc = reinterpret_cast<uint16_t *>(start + width);  // record: its column
    uint16_t *order = lc + kRound;                               // place in the round: its record
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int b = blockIdx.x;
    const int32_t p0 = __ldg(offsets + (int64_t)b * tiles);
    const int32_t p1 = b + 1 < buckets ? __ldg(offsets + (int64_t)(b + 1) * tiles) : (int32_t)nnz;
    const uint32_t cmask = (1u << bits.c) - 1u;
    const bool one = p1 - p0 <= kRound;
    if (!one) {
        for (int c = tid; c < width; c += kBucketThreads) next[c] = 0;
        __syncthreads();
        for (int32_t e = p0 + tid; e < p1; e += kBucketThreads)
            atomicAdd(next + (__ldg(reinterpret_cast<const uint32_t *>(rec + e)) & cmask), 1);
        __syncthreads();
        cta_scan<kBucketThreads>(next, width, sums);
    }
    bool first = true;
    for (int32_t q0 = p0; first || q0 < p1; q0 += kRound) {
        const int n = min(kRound, p1 - q0);
        for (int c = tid; c < width; c += kBucketThreads) start[c] = 0;
        if (tid == 0) n_long = 0;
        __syncthreads();
        for (int i = tid; i < n; i += 4 * kBucketThreads) {
            uint32_t k[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i + u * kBucketThreads < n)
                    k[u] = __ldg(reinterpret_cast<const uint32_t *>(rec + q0 + i + u * kBucketThreads)) & cmask;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i + u * kBucketThreads < n) {
                    lc[i + u * kBucketThreads] = (uint16_t)k[u];
                    atomicAdd(start + k[u], 1);
                }
        }
        __syncthreads();
        cta_scan<kBucketThreads>(start, width, sums);
        if (first) {
            for (int c = tid; c < width; c += kBucketThreads) {
                const int32_t at = p0 + (one ? start[c] : next[c]);
                next[c] = at;
                const int64_t column = (int64_t)b * width + c;
                if (column < n_cols) t_row_ptr[column] = at;
            }
            if (b == buckets - 1 && tid == 0) t_row_ptr[n_cols] = (int32_t)nnz;
            first = false;
            __syncthreads();
        }
        for (int i = tid; i < n; i += kBucketThreads) order[atomicAdd(start + lc[i], 1)] = (uint16_t)i;
        __syncthreads();
        // start[c] is now the end of column c, hence the start of column c + 1
        for (int c = tid; c < width; c += kBucketThreads) {
            const int s = c > 0 ? start[c - 1] : 0, m = start[c] - s;
            if (m > kShortColumn) {
                longs[atomicAdd(&n_long, 1)] = (int16_t)c;
                continue;
            }
            uint16_t *o = order + s;
            for (int i = 1; i < m; ++i) {
                const uint16_t v = o[i];
                int j = i;
                for (; j > 0 && o[j - 1] > v; --j) o[j] = o[j - 1];
                o[j] = v;
            }
        }
        __syncthreads();
        for (int l = wid; l < n_long; l += kBucketThreads / 32) {
            const int c = longs[l];
            int at = c > 0 ? start[c - 1] : 0;
            if (start[c] - at <= kRankColumn) {
                rank_places(order + at, start[c] - at);
                continue;
            }
            for (int i0 = 0; i0 < n; i0 += 32) {
                const bool in = i0 + lane < n && lc[i0 + lane] == c;
                const unsigned m = __ballot_sync(0xffffffffu, in);
                if (in) order[at + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(i0 + lane);
                at += __popc(m);
            }
        }
        __syncthreads();
        for (int i = tid; i < n; i += 4 * kBucketThreads) {
            int4 r[4];
            int c[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i + u * kBucketThreads < n) {
                    const int src = order[i + u * kBucketThreads];
                    c[u] = lc[src];
                    r[u] = __ldg(rec + q0 + src);
                }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i + u * kBucketThreads < n) {
                    const int32_t pos = next[c[u]] + (i + u * kBucketThreads) - (c[u] > 0 ? start[c[u] - 1] : 0);
                    const uint64_t key = rec_key(r[u]) >> bits.c;
                    T v;
                    rec_value(r[u], &v);
                    t_val[pos] = v;
                    t_col[pos] = (int32_t)(key >> bits.e);
                    tmap[pos] = (int32_t)(key & ((uint64_t(1) << bits.e) - 1));
                }
        }
        __syncthreads();
        for (int c = tid; c < width; c += kBucketThreads) next[c] += start[c] - (c > 0 ? start[c - 1] : 0);
        __syncthreads();
    }
}

// Buckets, tiles and workspace of a split.
struct SplitPlan {
    int width, buckets, seg;
    uint64_t magic;
    KeyBits bits;
    int64_t tiles;
    int64_t rec_bytes, count_bytes, scan_bytes;
    int64_t bytes() const { return 256 + rec_bytes + count_bytes + scan_bytes; }
};

// Dynamic shared memory of split_kernel and bucket_kernel.
static constexpr int split_smem_bytes(int buckets) { return (kSplitWarps * ((buckets + 1) / 2) + buckets) * 4; }
static constexpr int bucket_smem_bytes(int width) { return 8 * width + 4 * kRound; }

static int64_t align256(int64_t b) { return (b + 255) & ~int64_t(255); }

static int bits_for(uint64_t maxv) {
    int b = 0;
    while (b < 64 && (maxv >> b) != 0) ++b;
    return b;
}

// At most 2048 buckets (a tile's warps keep a counter for each in shared
// memory).  Within that, a bucket holds some 8192 entries (a round with room
// to spare), or fewer where that leaves SMs without a bucket; a tile is an
// eighth of an SM's share of the entries, at most 65,024.
static SplitPlan split_plan(const Mat &A) {
    SplitPlan p{};
    const int64_t want = std::max<int64_t>(256, std::min<int64_t>(8192, A.nnz / (num_sms() * 4)));
    const int64_t by_entries = (int64_t)((double)want * (double)A.n_cols / (double)A.nnz);
    p.width = (int)std::max<int64_t>(std::min<int64_t>(std::min<int64_t>(by_entries, A.n_cols), kMaxWidth),
                                     ceil_div(A.n_cols, kMaxBuckets));
    p.buckets = (int)ceil_div(A.n_cols, p.width);
    p.magic = ((uint64_t(1) << 40) + p.width - 1) / p.width;
    p.bits.c = bits_for((uint64_t)p.width - 1);
    p.bits.e = bits_for((uint64_t)A.nnz - 1);
    const int64_t share = ceil_div(A.nnz, (int64_t)num_sms() * 8 * kSplitWarps);
    p.seg = (int)std::max<int64_t>(32, std::min<int64_t>(ceil_div(share, 32) * 32, kSplitSegMax));
    p.tiles = ceil_div(A.nnz, (int64_t)kSplitWarps * p.seg);
    p.rec_bytes = align256(16 * A.nnz);
    p.count_bytes = align256(4 * p.buckets * p.tiles);
    p.scan_bytes = align256(scan_ws_bytes(p.buckets * p.tiles));
    return p;
}

// Every column must fall into one of at most 2048 buckets of 8192 columns,
// and a record's key into 64 bits.  Columns of 2^20 entries in the mean are
// too few buckets for the GPU, and a bucket is one CTA's, round after round:
// 8M entries in 1, 3 and 30 columns, split / radix sort: 27.9 / 5.3, 9.6 / 2.4
// and 1.2 / 1.8 ms.
bool transpose_split_fits(const Mat &A) {
    if (A.nnz <= 0 || A.n_cols > (int64_t)kMaxBuckets * kMaxWidth || A.nnz >> 20 >= A.n_cols) return false;
    const SplitPlan p = split_plan(A);
    return p.bits.c + p.bits.e + bits_for((uint64_t)A.n_rows - 1) <= 64;
}

int64_t transpose_split_bytes(const Mat &A) { return split_plan(A).bytes(); }

template <typename T>
static gbsp_status split_build(const Mat &A, const gbsp_transpose_buffers &b, cudaStream_t s) {
    const SplitPlan p = split_plan(A);
    // records on a 16-byte boundary, wherever the caller's workspace starts
    char *w = reinterpret_cast<char *>((reinterpret_cast<uintptr_t>(b.workspace) + 255) & ~uintptr_t(255));
    int4 *rec = reinterpret_cast<int4 *>(w);
    w += p.rec_bytes;
    int32_t *counts = reinterpret_cast<int32_t *>(w);
    w += p.count_bytes;
    int32_t *scan_ws = reinterpret_cast<int32_t *>(w);
    int32_t *row_of = b.t_col;  // each entry's row, until level 2 writes t_col
    row_of_launch(A, row_of, s);
    split_count_kernel<<<(unsigned)p.tiles, kSplitThreads, 0, s>>>(A.nnz, p.magic, p.buckets, p.tiles,
                                                                   (int64_t)kSplitWarps * p.seg, A.col, counts);
    GBSP_LAUNCH_CHECK("split_count_kernel");
    gbsp_status st = scan_exclusive(counts, p.buckets * p.tiles, counts, nullptr, scan_ws, s);
    if (st != GBSP_OK) return st;
    const int smem = split_smem_bytes(p.buckets);
    GBSP_SMEM_LIMIT(split_kernel<T>, split_smem_bytes(kMaxBuckets));
    split_kernel<T><<<(unsigned)p.tiles, kSplitThreads, smem, s>>>(A.nnz, p.width, p.magic, p.bits, p.buckets, p.tiles,
                                                                   p.seg, A.col, row_of, static_cast<const T *>(A.val),
                                                                   counts, rec);
    GBSP_LAUNCH_CHECK("split_kernel");
    const int bsmem = bucket_smem_bytes(p.width);
    GBSP_SMEM_LIMIT(bucket_kernel<T>, bucket_smem_bytes(kMaxWidth));
    bucket_kernel<T><<<(unsigned)p.buckets, kBucketThreads, bsmem, s>>>(A.n_cols, A.nnz, p.width, p.bits, p.buckets,
                                                                        p.tiles, counts, rec, b.t_row_ptr, b.t_col,
                                                                        static_cast<T *>(b.t_val), b.tmap);
    GBSP_LAUNCH_CHECK("bucket_kernel");
    return GBSP_OK;
}

gbsp_status transpose_split_build(const Mat &A, const gbsp_transpose_buffers &b, cudaStream_t s) {
    return A.dtype == GBSP_F64 ? split_build<double>(A, b, s) : split_build<float>(A, b, s);
}

}  // namespace gbsp
