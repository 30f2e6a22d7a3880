// Row lookup shared by the kernels that walk CRS entries 32 at a time.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gbsp {

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

}  // namespace gbsp
