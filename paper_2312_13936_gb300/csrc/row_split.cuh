// Rows too long for a block's shared memory, split by ranges of their targets
// so that what remains to be sorted is short, or dense enough in its range
// that a bitmap of the range is no longer than it. (A bitmap over all vertices
// for every such row, walked by one block, cost with the graph's vertices
// instead of the row's entries. Edge lists, ms a call: 300 rows of 17,000
// entries among 3e8 vertices 360, by ranges 38; among 3e7, 22.2 and 10.3; R-MAT
// of 2^24 vertices, 40 edges a vertex, 303 and 161; up to 2^20 vertices, where
// the rows stay whole, the same. Deterministic aggregation of R-MAT of 2^23
// vertices 247 and 201 ms.)
#pragma once
#include "common.cuh"

namespace lgb {

// Splits the rows rows[0, gridDim.x) by target >> bits into nr parts each, part
// p nr + r holding row p's targets of range r. Each row, of the entries
// [off[row], off[row] + deg[row]) (deg null: to off[row + 1]), is shared by
// gridDim.y blocks, which count their share in shared memory first (nr words;
// 3 nr with PLACE), so that a part's counter takes one atomic a block.
// !PLACE: cnt[part] += its entries. PLACE: entries to start[part] and on (in no
// particular order), cnt zero before.
template <class W, bool PLACE>
__global__ void __launch_bounds__(256) k_split_rows(const int32_t *__restrict__ rows, const int64_t *__restrict__ off,
                                                    const int32_t *__restrict__ deg, const int32_t *__restrict__ tgt,
                                                    const W *__restrict__ w, int bits, int nr,
                                                    unsigned long long *cnt, const int64_t *__restrict__ start,
                                                    int32_t *tgt2, W *w2) {
    extern __shared__ __align__(8) unsigned char smem[];
    int64_t *base = reinterpret_cast<int64_t *>(smem);                        // PLACE
    int32_t *own = reinterpret_cast<int32_t *>(smem + (PLACE ? 8 * (size_t)nr : 0));
    const int32_t r = rows[blockIdx.x];
    const int64_t o = off[r], d = deg ? (int64_t)deg[r] : off[r + 1] - o;
    const int64_t part0 = (int64_t)blockIdx.x * nr;
    const int64_t first = (int64_t)blockIdx.y * blockDim.x + threadIdx.x, step = (int64_t)gridDim.y * blockDim.x;
    for (int b = threadIdx.x; b < nr; b += blockDim.x) own[b] = 0;
    __syncthreads();
    for (int64_t e = first; e < d; e += step) atomicAdd(&own[tgt[o + e] >> bits], 1);
    __syncthreads();
    for (int b = threadIdx.x; b < nr; b += blockDim.x) {
        const int32_t c = own[b];
        if (c == 0) continue;
        const unsigned long long at = atomicAdd(&cnt[part0 + b], (unsigned long long)c);
        if (PLACE) {
            base[b] = start[part0 + b] + (int64_t)at;
            own[b] = 0;
        }
    }
    if (!PLACE) return;
    __syncthreads();
    for (int64_t e = first; e < d; e += step) {
        const int32_t k = tgt[o + e];
        const int64_t at = base[k >> bits] + atomicAdd(&own[k >> bits], 1);
        tgt2[at] = k;
        if (w) w2[at] = w[o + e];
    }
}
inline size_t split_smem(int nr, bool place) { return (size_t)nr * (place ? 12 : 4); }

}  // namespace lgb
