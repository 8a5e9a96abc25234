// Edge list to symmetric CSR on the GPU: the input preparation of the
// paper's experiments (edges made undirected, reverse edges added, unit
// weight by default; Section 5.1, Table 2). Every edge (u, v) with u != v
// gives the entries (u, v) and (v, u); a self-loop gives one entry (reading
// R11) unless dropped. Entries are counted per row and scattered into row
// segments (a counting sort by row, with 64-bit positions, so edge lists of
// billions of edges fit); then every row is sorted by target by itself and
// its entries with equal targets are merged (weights summed in fp64 and
// rounded once, or the largest kept) at the front of its segment: rows of up
// to 32 entries by a tile of lanes, of up to 256 by a warp, of up to kRowSmem
// by a block in shared memory. Row offsets come from a scan of the merged row
// lengths, and the fronts are copied to their places. Longer rows are split by
// ranges of kRangeBits target bits (row_split.cuh) into parts that are sorted
// and merged as rows are; a part longer than kRowSmem is not sorted: a bitmap
// of its range, no longer than twice its entries, counts its targets, and the
// running population count is every target's place. (Sorting all entries by (row, target) with
// 8-bit digits moved them six times at a million vertices, some 50 bytes an
// entry and digit: 24 of 28.5 ms for 47M edges.)
#include <cmath>
#include <string>
#include <utility>
#include <vector>

#include "common.cuh"
#include "engine.h"
#include "kernels.h"
#include "row_split.cuh"

namespace lgb {
namespace {

constexpr int kRowWarp = 256;
constexpr int kRowSmem = 16384;  // 12 bytes an entry of shared memory and the buckets
constexpr int64_t kMaxRow = (int64_t)1 << 30;
constexpr int kBigSplit = 32;    // blocks that share a row of more than kRowSmem entries
constexpr int kRangeBits = 20;   // a range's bitmap and counts are 2 x 32,768 words
constexpr int64_t kBitmapBytes = (int64_t)1 << 31;  // bitmaps and their counts, for the long parts taken at once
constexpr int kRowBins = 6;      // 1: up to 8 entries, 2: 32, 3: kRowWarp, 4: 2048, 5: kRowSmem, 6: longer (0 unused)

inline int grid_for(int64_t n, int threads) {
    int64_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    return (int)(b > 152 * 16 ? 152 * 16 : b);
}
#define GRID_STRIDE(i, n) \
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (n); i += (int64_t)gridDim.x * blockDim.x)

// entries per row: row u counts (u, v), row v counts (v, u) for u != v; a
// self-loop counts once unless dropped. err = 1 for an endpoint outside
// [0, n) or a weight that is not finite and >= 0 (such an edge is skipped).
__global__ void k_count_rows(int64_t n, int64_t m, const int32_t *src, const int32_t *dst, const float *w,
                             int drop_self, unsigned long long *cnt, int *err) {
    GRID_STRIDE(e, m) {
        const int32_t u = src[e], v = dst[e];
        const float x = w ? w[e] : 1.0f;
        if (!(u >= 0 && u < n && v >= 0 && v < n && isfinite(x) && x >= 0.0f)) {
            set_error(err, 1);
            continue;
        }
        if (u != v) {
            atomicAdd(&cnt[u], 1ULL);
            atomicAdd(&cnt[v], 1ULL);
        } else if (!drop_self) {
            atomicAdd(&cnt[u], 1ULL);
        }
    }
}
// scatter every entry into its row segment (the targets of a row in no
// particular order)
__global__ void k_scatter_rows(int64_t m, const int32_t *src, const int32_t *dst, const float *w, int drop_self,
                               const int64_t *rowstart, unsigned long long *cursor, int32_t *tgt, float *wt) {
    GRID_STRIDE(e, m) {
        const int32_t u = src[e], v = dst[e];
        if (u == v && drop_self) continue;
        const float x = wt ? w[e] : 1.0f;
        const int64_t p = rowstart[u] + (int64_t)atomicAdd(&cursor[u], 1ULL);
        tgt[p] = v;
        if (wt) wt[p] = x;
        if (u != v) {
            const int64_t q = rowstart[v] + (int64_t)atomicAdd(&cursor[v], 1ULL);
            tgt[q] = u;
            if (wt) wt[q] = x;
        }
    }
}
__global__ void k_row_bins(const int64_t *rowstart, int64_t n, int32_t *bin) {
    GRID_STRIDE(r, n) {
        const int64_t d = rowstart[r + 1] - rowstart[r];
        bin[r] = d <= 0 ? -1 : d <= 8 ? 1 : d <= 32 ? 2 : d <= kRowWarp ? 3 : d <= 2048 ? 4 : d <= kRowSmem ? 5 : 6;
    }
}

__device__ __forceinline__ double combined(double s, double x, int combine) { return combine ? fmax(s, x) : s + x; }

// T lanes per row of up to T entries: equal targets find one another with one
// match, the first lane of each keeps the merged weight, and its place is the
// number of first lanes with smaller targets.
template <int T>
__global__ void __launch_bounds__(256) k_row_tile(const int32_t *__restrict__ list, int64_t count,
                                                  const int64_t *__restrict__ rowstart, int32_t *tgt, float *wt,
                                                  float *mw, int combine, int64_t *rowlen) {
    const int lane = threadIdx.x & 31, tl = lane & (T - 1), base = lane & ~(T - 1);
    const unsigned tmask = T == 32 ? kFull : ((1u << T) - 1u) << base;
    const int64_t tiles = (int64_t)gridDim.x * (blockDim.x / T);
    for (int64_t t = (int64_t)blockIdx.x * (blockDim.x / T) + threadIdx.x / T; t < count; t += tiles) {
        const int32_t r = list[t];
        const int64_t o = rowstart[r];
        const int d = (int)(rowstart[r + 1] - o);
        const int32_t k = tl < d ? tgt[o + tl] : -1;
        const float x = (wt && tl < d) ? wt[o + tl] : 1.0f;
        const unsigned peers = __match_any_sync(tmask, k);
        const bool head = k >= 0 && __ffs(peers) - 1 == lane;
        const int32_t mine = head ? k : INT32_MAX;
        int pos = 0;
#pragma unroll
        for (int j = 0; j < T; ++j) pos += __shfl_sync(tmask, mine, j, T) < mine ? 1 : 0;
        double s = wt ? (double)x : (combine ? 1.0 : (double)__popc(peers));
        if (wt && __any_sync(tmask, k >= 0 && !head)) {
            for (int j = 0; j < T; ++j) {
                const float y = __shfl_sync(tmask, x, j, T);
                if (head && base + j != lane && (peers >> (base + j) & 1u)) s = combined(s, (double)y, combine);
            }
        }
        const unsigned heads = __ballot_sync(tmask, head) & tmask;
        if (head) {
            tgt[o + pos] = k;
            mw[o + pos] = (float)s;
        }
        if (tl == 0) rowlen[r] = __popc(heads);
    }
}

// A warp per row of up to kRowWarp entries: the lanes count each target's
// smaller ones (equal ones by place) for its place in order, and the sorted
// targets, in shared memory, are merged by neighbour.
__global__ void __launch_bounds__(256) k_row_warp(const int32_t *__restrict__ list, int64_t count,
                                                  const int64_t *__restrict__ rowstart, int32_t *tgt, float *wt,
                                                  float *mw, int combine, int64_t *rowlen) {
    __shared__ __align__(16) int32_t s_key[8][kRowWarp];
    __shared__ float s_w[8][kRowWarp];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    int32_t *key = s_key[wib];
    float *sw = s_w[wib];
    const int64_t warps = (int64_t)gridDim.x * 8;
    for (int64_t t = (int64_t)blockIdx.x * 8 + wib; t < count; t += warps) {
        const int32_t r = list[t];
        const int64_t o = rowstart[r];
        const int d = (int)(rowstart[r + 1] - o), pad = (d + 3) & ~3, n = (d + 31) / 32;
        int32_t k[8], rank[8];
        float x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int e = q * 32 + lane;
            k[q] = INT32_MAX;
            x[q] = 1.0f;
            rank[q] = 0;
            if (e < d) {
                k[q] = tgt[o + e];
                if (wt) x[q] = wt[o + e];
            }
            if (e < pad) key[e] = k[q];
        }
        __syncwarp();
        for (int e = 0; e < pad; e += 4) {
            const int4 y = *reinterpret_cast<const int4 *>(&key[e]);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q < n) {
                    const int p = q * 32 + lane;  // an equal target before this one counts as smaller
                    rank[q] += (y.x < k[q] + (e < p)) + (y.y < k[q] + (e + 1 < p)) + (y.z < k[q] + (e + 2 < p)) +
                               (y.w < k[q] + (e + 3 < p));
                }
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (q * 32 + lane < d) {
                key[rank[q]] = k[q];
                sw[rank[q]] = x[q];
            }
        __syncwarp();
        int done = 0;
        for (int e0 = 0; e0 < d; e0 += 32) {
            const int e = e0 + lane;
            const bool head = e < d && (e == 0 || key[e] != key[e - 1]);
            const unsigned heads = __ballot_sync(kFull, head);
            if (head) {
                double s = (double)sw[e];
                for (int j = e + 1; j < d && key[j] == key[e]; ++j) s = combined(s, (double)sw[j], combine);
                const int64_t at = o + done + __popc(heads & ((1u << lane) - 1u));
                tgt[at] = key[e];
                mw[at] = (float)s;
            }
            done += __popc(heads);
        }
        if (lane == 0) rowlen[r] = done;
        __syncwarp();
    }
}

// A block per row of up to cap entries, in shared memory: a counting sort by
// the targets' high bits (bucket = (target & mask) >> shift; the bits above mask
// are the same in the whole row), then every entry counts
// the smaller targets of its own bucket -- a handful, since a bucket holds few
// of a row's targets -- for its place in order, and equal neighbours are
// merged, every thread a run of consecutive ones. (A bitonic network of
// (target, place) words took 66 to 105 rounds of the block: 5.3 of 10 ms for
// 47M edges.) A row whose targets crowd into few buckets -- neighbours close
// by in a graph of many vertices, one edge listed over and over -- would
// compare every entry with hundreds or thousands, up to the square of the row:
// beyond kRowCrowd comparisons an entry on average the network is the shorter
// way, and its work does not depend on the targets.
constexpr int kRowBuckets = 2048;
constexpr int kRowCrowd = 256;
__global__ void __launch_bounds__(512) k_row_block(const int32_t *__restrict__ list, int64_t count,
                                                   const int64_t *__restrict__ rowstart, int32_t *tgt, float *wt,
                                                   float *mw, int combine, int64_t *rowlen, int cap, int32_t mask,
                                                   int shift) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_part[16];
    int32_t *raw = reinterpret_cast<int32_t *>(smem);      // by bucket
    int32_t *key = raw + cap;                              // in order
    float *x = reinterpret_cast<float *>(key + cap);       // weights by bucket, then in order (one array:
                                                           // a thread's own entries pass through registers)
    int32_t *end = reinterpret_cast<int32_t *>(x + cap);   // a bucket's cursor, at last its end
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5, nw = blockDim.x >> 5;
    // exclusive scan of the threads' values; *all the block's sum
    auto block_scan = [&](int v, int *all) {
        int inc = v;
        for (int q = 1; q < 32; q <<= 1) {
            const int y = __shfl_up_sync(kFull, inc, q);
            if (lane >= q) inc += y;
        }
        __syncthreads();
        if (lane == 31) s_part[wib] = inc;
        __syncthreads();
        int before = inc - v, sum = 0;
        for (int q = 0; q < nw; ++q) {
            if (q < wib) before += s_part[q];
            sum += s_part[q];
        }
        *all = sum;
        return before;
    };
    constexpr int kPer = kRowSmem / 512;  // entries of a thread
    for (int64_t t = blockIdx.x; t < count; t += gridDim.x) {
        const int32_t r = list[t];
        const int64_t o = rowstart[r];
        const int d = (int)(rowstart[r + 1] - o);
        int all;
        for (int b = tid; b < kRowBuckets; b += blockDim.x) end[b] = 0;
        __syncthreads();
        for (int e = tid; e < d; e += blockDim.x) {
            const int32_t k = tgt[o + e];
            key[e] = k;
            atomicAdd(&end[(k & mask) >> shift], 1);
        }
        __syncthreads();
        int crowd = 0;  // comparisons of the row: every bucket's square
        {
            constexpr int own = kRowBuckets / 256;  // of a thread, in 256 threads
            int c[own], sum = 0, sq = 0;
            for (int q = 0; q < own; ++q) {
                c[q] = tid < 256 ? end[tid * own + q] : 0;
                sum += c[q];
                sq += c[q] * c[q];
            }
            block_scan(sq, &crowd);
            int run = block_scan(sum, &all);
            for (int q = 0; q < own; ++q)
                if (tid < 256) {
                    end[tid * own + q] = run;
                    run += c[q];
                }
        }
        __syncthreads();
        float keep[kPer];
        int place[kPer];
        if (crowd <= d * kRowCrowd) {
            for (int e = tid; e < d; e += blockDim.x) {
                const int32_t k = key[e];
                const int at = atomicAdd(&end[(k & mask) >> shift], 1);
                raw[at] = k;
                x[at] = wt ? wt[o + e] : 1.0f;
            }
            __syncthreads();
            for (int q = 0, e = tid; q < kPer; ++q, e += blockDim.x) {
                if (e >= d) break;
                const int32_t k = raw[e];
                const int b = (k & mask) >> shift, lo = b > 0 ? end[b - 1] : 0, hi = end[b];
                int rank = lo;
                for (int j = lo; j < hi; ++j) rank += raw[j] < k + (j < e);  // an equal one before counts as smaller
                keep[q] = x[e];
                place[q] = rank;
            }
            __syncthreads();
            for (int q = 0, e = tid; q < kPer; ++q, e += blockDim.x) {
                if (e >= d) break;
                key[place[q]] = raw[e];
                x[place[q]] = keep[q];
            }
            __syncthreads();
        } else {
            unsigned long long *word = reinterpret_cast<unsigned long long *>(smem);  // over raw and key
            int P = 32;
            while (P < d) P <<= 1;
            for (int e = tid; e < P; e += blockDim.x) {
                word[e] = e < d ? ((unsigned long long)(uint32_t)tgt[o + e] << 32) | (uint32_t)e : ~0ULL;
                if (e < d) x[e] = wt ? wt[o + e] : 1.0f;
            }
            __syncthreads();
            for (int size = 2; size <= P; size <<= 1)
                for (int st = size >> 1; st > 0; st >>= 1) {
                    for (int i = tid; i < P / 2; i += blockDim.x) {
                        const int lo = 2 * i - (i & (st - 1));
                        const unsigned long long p = word[lo], q = word[lo + st];
                        if ((p > q) == ((lo & size) == 0)) {
                            word[lo] = q;
                            word[lo + st] = p;
                        }
                    }
                    __syncthreads();
                }
            for (int q = 0, e = tid; q < kPer; ++q, e += blockDim.x) {
                if (e >= d) break;
                place[q] = (int)(word[e] >> 32);
                keep[q] = x[(uint32_t)word[e]];
            }
            __syncthreads();
            for (int q = 0, e = tid; q < kPer; ++q, e += blockDim.x) {
                if (e >= d) break;
                key[e] = place[q];
                x[e] = keep[q];
            }
            __syncthreads();
        }
        const int per = (d + blockDim.x - 1) / blockDim.x, e0 = min(d, tid * per), e1 = min(d, e0 + per);
        int heads = 0;
        for (int e = e0; e < e1; ++e) heads += e == 0 || key[e] != key[e - 1];
        int at = block_scan(heads, &all);
        for (int e = e0; e < e1; ++e) {
            const int32_t k = key[e];
            if (e > 0 && k == key[e - 1]) continue;
            double s = (double)x[e];
            for (int j = e + 1; j < d && key[j] == k; ++j) s = combined(s, (double)x[j], combine);
            tgt[o + at] = k;
            mw[o + at] = (float)s;
            ++at;
        }
        if (tid == 0) rowlen[r] = all;
        __syncthreads();
    }
}

// ---- rows (or parts) of more than kRowSmem entries, their targets the same
// above mask: rows [p0, p0 + gridDim.x) of list
__global__ void k_long_set(const int32_t *list, int64_t p0, const int64_t *rowstart, const int32_t *tgt, int32_t mask,
                           unsigned *bits, int64_t nwords) {
    const int32_t r = list[p0 + blockIdx.x];
    const int64_t o = rowstart[r], d = rowstart[r + 1] - o;
    unsigned *m = bits + (int64_t)blockIdx.x * nwords;
    for (int64_t e = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; e < d; e += (int64_t)gridDim.y * blockDim.x) {
        const int32_t k = tgt[o + e] & mask;
        atomicOr(&m[k >> 5], 1u << (k & 31));
    }
}
// targets before each word of a row's bitmap, and the row's merged length
__global__ void __launch_bounds__(1024) k_long_count(const int32_t *list, int64_t p0, const unsigned *bits,
                                                     unsigned *before, int64_t nwords, int64_t *rowlen) {
    __shared__ unsigned s_w[32];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const unsigned *m = bits + (int64_t)blockIdx.x * nwords;
    unsigned *out = before + (int64_t)blockIdx.x * nwords;
    unsigned carry = 0;
    for (int64_t i0 = 0; i0 < nwords; i0 += blockDim.x) {
        const int64_t i = i0 + threadIdx.x;
        const unsigned own = i < nwords ? __popc(m[i]) : 0;
        unsigned inc = own;
        for (int q = 1; q < 32; q <<= 1) {
            const unsigned y = __shfl_up_sync(kFull, inc, q);
            if (lane >= q) inc += y;
        }
        if (lane == 31) s_w[wib] = inc;
        __syncthreads();
        unsigned mine = carry, all = 0;
        for (int q = 0; q < 32; ++q) {
            if (q < wib) mine += s_w[q];
            all += s_w[q];
        }
        if (i < nwords) out[i] = mine + inc - own;
        carry += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) rowlen[list[p0 + blockIdx.x]] = carry;
}
// every entry to its target's place: the target to the output, its weight
// into the place's fp64 sum (or maximum) acc, which holds the places of the
// rows taken at once (row p at abase[p - p0])
__global__ void k_long_place(const int32_t *list, int64_t p0, const int64_t *rowstart, const int32_t *tgt,
                             const float *wt, int combine, int32_t mask, const unsigned *bits, const unsigned *before,
                             int64_t nwords, const int64_t *place, int32_t *idx, double *acc, const int64_t *abase) {
    const int32_t r = list[p0 + blockIdx.x];
    const int64_t o = rowstart[r], d = rowstart[r + 1] - o, out = place[r];
    const unsigned *m = bits + (int64_t)blockIdx.x * nwords, *f = before + (int64_t)blockIdx.x * nwords;
    double *s = acc + abase[blockIdx.x];
    for (int64_t e = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; e < d; e += (int64_t)gridDim.y * blockDim.x) {
        const int32_t k = tgt[o + e];
        const int32_t x5 = (k & mask) >> 5;
        const int64_t at = f[x5] + __popc(m[x5] & ((1u << (k & 31)) - 1u));
        idx[out + at] = k;
        const double x = wt ? (double)wt[o + e] + 0.0 : 1.0;  // (no -0.0)
        if (combine)  // weights are not negative: their bits are ordered as they are
            atomicMax(reinterpret_cast<unsigned long long *>(&s[at]), (unsigned long long)__double_as_longlong(x));
        else
            atomicAdd(&s[at], x);
    }
}
__global__ void k_long_weights(const int32_t *list, int64_t p0, const int64_t *place, const int64_t *rowlen,
                               const double *acc, const int64_t *abase, float *w) {
    const int32_t r = list[p0 + blockIdx.x];
    const int64_t o = place[r], d = rowlen[r];
    const double *s = acc + abase[blockIdx.x];
    for (int64_t e = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; e < d; e += (int64_t)gridDim.y * blockDim.x)
        w[o + e] = (float)s[e];
}

__global__ void k_long_lens(const int32_t *list, int64_t p0, int64_t c, const int64_t *rowlen, int64_t *lens) {
    GRID_STRIDE(k, c) lens[k] = rowlen[list[p0 + k]];
}

// ---- parts of the split rows list[0, nrows), nr each; so: scan of their merged
// lengths
__global__ void k_part_rows(const int32_t *list, int64_t nrows, int nr, const int64_t *so, int64_t *rowlen) {
    GRID_STRIDE(p, nrows) rowlen[list[p]] = so[(p + 1) * nr] - so[p * nr];
}
// place of every part in the output
__global__ void k_part_places(const int32_t *list, int64_t nparts, int nr, const int64_t *so, const int64_t *off,
                              int64_t *place) {
    GRID_STRIDE(k, nparts) {
        const int64_t p = k / nr;
        place[k] = off[list[p]] + so[k] - so[p * nr];
    }
}

// the merged front of every row (or part) of the list to its place in the
// output: T lanes a row
template <int T>
__global__ void __launch_bounds__(256) k_row_copy(const int32_t *__restrict__ list, int64_t count,
                                                  const int64_t *__restrict__ rowstart,
                                                  const int64_t *__restrict__ rowlen,
                                                  const int64_t *__restrict__ place, const int32_t *tgt,
                                                  const float *mw, int32_t *idx, float *w) {
    const int tl = threadIdx.x & (T - 1);
    const int64_t tiles = (int64_t)gridDim.x * (blockDim.x / T);
    for (int64_t t = (int64_t)blockIdx.x * (blockDim.x / T) + threadIdx.x / T; t < count; t += tiles) {
        const int32_t r = list[t];
        const int64_t s = rowstart[r], o = place[r], d = rowlen[r];
        for (int64_t e = tl; e < d; e += T) {
            idx[o + e] = tgt[s + e];
            w[o + e] = mw[s + e];
        }
    }
}

// rows (or parts of rows), each a segment of entries, merged at its front
struct Segments {
    const int64_t *start = nullptr;  // and one more
    int32_t *tgt = nullptr;
    float *wt = nullptr, *mw = nullptr;  // weights (null: ones), merged ones
    int64_t *len = nullptr;              // merged lengths
    int32_t *list = nullptr;             // by length: bin b at [hb[b], hb[b + 1])
    int64_t hb[kRowBins + 2] = {0};
    int64_t count(int b) const { return hb[b + 1] - hb[b]; }
};

// every segment of bins 1 to 5 sorted and merged; none is longer than longest,
// and the targets of each agree above mask
cudaError_t sort_segments(const Segments &g, int64_t longest, int32_t mask, int combine, cudaStream_t s) {
    if (const int64_t c = g.count(1))
        k_row_tile<8><<<grid_for(c, 32), 256, 0, s>>>(g.list + g.hb[1], c, g.start, g.tgt, g.wt, g.mw, combine, g.len);
    if (const int64_t c = g.count(2))
        k_row_tile<32><<<grid_for(c, 8), 256, 0, s>>>(g.list + g.hb[2], c, g.start, g.tgt, g.wt, g.mw, combine, g.len);
    if (const int64_t c = g.count(3))
        k_row_warp<<<grid_for(c, 8), 256, 0, s>>>(g.list + g.hb[3], c, g.start, g.tgt, g.wt, g.mw, combine, g.len);
    auto block_bytes = [](int c) { return (size_t)c * 12 + 4 * kRowBuckets; };
    int shift = 0;  // the targets' bits under mask into kRowBuckets buckets
    while ((mask >> shift) >= kRowBuckets) ++shift;
    cudaError_t e = cudaFuncSetAttribute(k_row_block, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)block_bytes(kRowSmem));
    if (e != cudaSuccess) return e;
    if (const int64_t c = g.count(4))
        k_row_block<<<grid_for(c, 1), 256, block_bytes(2048), s>>>(g.list + g.hb[4], c, g.start, g.tgt, g.wt, g.mw,
                                                                   combine, g.len, 2048, mask, shift);
    if (const int64_t c = g.count(5)) {
        int cap = 4096;
        while (cap < longest && cap < kRowSmem) cap <<= 1;
        k_row_block<<<grid_for(c, 1), 512, block_bytes(cap), s>>>(g.list + g.hb[5], c, g.start, g.tgt, g.wt, g.mw,
                                                                  combine, g.len, cap, mask, shift);
    }
    return cudaGetLastError();
}
// the merged fronts of bins 1 to 5 to their places
cudaError_t copy_segments(const Segments &g, const int64_t *place, int32_t *idx, float *w, cudaStream_t s) {
    const int64_t c1 = g.count(1), c2 = g.hb[6] - g.hb[2];
    if (c1 > 0)
        k_row_copy<8><<<grid_for(c1, 32), 256, 0, s>>>(g.list + g.hb[1], c1, g.start, g.len, place, g.tgt, g.mw, idx, w);
    if (c2 > 0)
        k_row_copy<32><<<grid_for(c2, 8), 256, 0, s>>>(g.list + g.hb[2], c2, g.start, g.len, place, g.tgt, g.mw, idx, w);
    return cudaGetLastError();
}

}  // namespace

leiden_status csr_from_edges(int64_t n, int64_t m, const int32_t *src, const int32_t *dst, const float *w, int where,
                             int drop_self, int combine, int64_t *offsets, int32_t *indices, float *weights,
                             int64_t *nnz_io, cudaStream_t s) {
    if (n < 0 || n > INT32_MAX || m < 0 || !nnz_io || !offsets || (m > 0 && (!src || !dst)) ||
        (where != LEIDEN_HOST && where != LEIDEN_DEVICE) || (combine != 0 && combine != 1)) {
        set_last_error("leiden_csr_from_edges: invalid arguments");
        return LEIDEN_ERR_INVALID;
    }
    const int64_t cap = *nnz_io;
    std::vector<void *> mem;
    auto get = [&](void **p, size_t bytes) -> bool {
        if (cudaMallocAsync(p, bytes ? bytes : 1, s) != cudaSuccess) return false;
        mem.push_back(*p);
        return true;
    };
    auto release = [&]() {
        for (void *p : mem) cudaFreeAsync(p, s);
        mem.clear();
    };
    auto fail = [&](leiden_status st, const std::string &msg) {
        release();
        set_last_error(msg);
        return st;
    };
    cudaError_t e = cudaSuccess;
#define IK(x)                                                                                        \
    do {                                                                                             \
        if ((e = (x)) != cudaSuccess) return fail(LEIDEN_ERR_CUDA, std::string("leiden_csr_from_edges: ") + \
                                                  cudaGetErrorString(e));                           \
    } while (0)
    const cudaMemcpyKind in_kind = where == LEIDEN_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
    const cudaMemcpyKind out_kind = where == LEIDEN_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
    const int32_t *dsrc = src, *ddst = dst;
    const float *dw = w;
    unsigned long long *cnt = nullptr;
    int64_t *rowstart = nullptr, *doff = nullptr, *rowlen = nullptr;
    int *err = nullptr;
    void *scan_tmp = nullptr;
    if (!get((void **)&cnt, 8 * (size_t)(n + 1)) || !get((void **)&rowstart, 8 * (size_t)(n + 1)) ||
        !get((void **)&rowlen, 8 * (size_t)(n + 1)) || !get((void **)&doff, 8 * (size_t)(n + 1)) ||
        !get((void **)&err, sizeof(int)) || !get(&scan_tmp, scan_tmp_bytes(n + 1)))
        return fail(LEIDEN_ERR_OOM, "leiden_csr_from_edges: device allocation failed");
    if (where == LEIDEN_HOST && m > 0) {  // the edge list on the device
        int32_t *a = nullptr, *b = nullptr;
        float *c = nullptr;
        if (!get((void **)&a, 4 * (size_t)m) || !get((void **)&b, 4 * (size_t)m) || (w && !get((void **)&c, 4 * (size_t)m)))
            return fail(LEIDEN_ERR_OOM, "leiden_csr_from_edges: device allocation failed");
        IK(cudaMemcpyAsync(a, src, 4 * (size_t)m, in_kind, s));
        IK(cudaMemcpyAsync(b, dst, 4 * (size_t)m, in_kind, s));
        if (w) IK(cudaMemcpyAsync(c, w, 4 * (size_t)m, in_kind, s));
        dsrc = a;
        ddst = b;
        dw = c;
    }
    // ---- entries per row, row starts, the longest row
    unsigned long long *longest = nullptr;
    if (!get((void **)&longest, 8)) return fail(LEIDEN_ERR_OOM, "leiden_csr_from_edges: device allocation failed");
    IK(cudaMemsetAsync(err, 0, sizeof(int), s));
    IK(cudaMemsetAsync(cnt, 0, 8 * (size_t)(n + 1), s));
    IK(cudaMemsetAsync(rowlen, 0, 8 * (size_t)(n + 1), s));
    if (m > 0) {
        k_count_rows<<<grid_for(m, 256), 256, 0, s>>>(n, m, dsrc, ddst, dw, drop_self, cnt, err);
        IK(cudaGetLastError());
    }
    IK(launch_exclusive_scan(reinterpret_cast<const int64_t *>(cnt), rowstart, n, scan_tmp, s));
    IK(launch_max_i64(reinterpret_cast<const int64_t *>(cnt), n, longest, s));
    int herr = 0;
    int64_t M = 0;  // entries before merging
    unsigned long long hlongest = 0;
    IK(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s));
    IK(cudaMemcpyAsync(&M, rowstart + n, 8, cudaMemcpyDeviceToHost, s));
    IK(cudaMemcpyAsync(&hlongest, longest, 8, cudaMemcpyDeviceToHost, s));
    IK(cudaStreamSynchronize(s));
    if (herr) return fail(LEIDEN_ERR_INVALID, "leiden_csr_from_edges: endpoint outside [0, n) or bad weight");
    if ((int64_t)hlongest > kMaxRow)
        return fail(LEIDEN_ERR_INVALID, "leiden_csr_from_edges: a row of more than 2^30 entries before merging");
    int64_t nnz = 0;
    int32_t *sti = indices;
    float *stw = weights;
    Segments rows, parts;        // of the long rows (more than one range)
    const Segments *lg = &rows;  // whose bin 6 goes through bitmaps
    int32_t lmask = INT32_MAX;
    int64_t nwords = (n + 31) / 32, nrange = 1, nlong = 0, nparts = 0, at_once = 0;
    unsigned *bits = nullptr, *before = nullptr;
    int64_t *abase = nullptr, *so = nullptr, *place = nullptr;
    const int64_t *lplace = doff;
    // segments by length
    auto bins = [&](Segments &g, int64_t count, const int64_t *start) -> leiden_status {
        int32_t *bin = nullptr;
        int64_t *bin_off = nullptr;
        void *part_tmp = nullptr;
        if (!get((void **)&bin, 4 * (size_t)count) || !get((void **)&g.list, 4 * (size_t)count) ||
            !get((void **)&bin_off, 8 * (kRowBins + 2)) || !get(&part_tmp, partition_tmp_bytes(count, kRowBins + 1)))
            return fail(LEIDEN_ERR_OOM, "leiden_csr_from_edges: device allocation failed");
        g.start = start;
        k_row_bins<<<grid_for(count, 256), 256, 0, s>>>(start, count, bin);
        IK(cudaGetLastError());
        IK(launch_partition(bin, count, kRowBins + 1, bin_off, g.list, part_tmp, s));
        IK(cudaMemcpyAsync(g.hb, bin_off, 8 * (kRowBins + 2), cudaMemcpyDeviceToHost, s));
        IK(cudaStreamSynchronize(s));
        return LEIDEN_OK;
    };
    leiden_status st = LEIDEN_OK;
    if (M > 0) {
        // ---- scatter into row segments; rows by length
        if (!get((void **)&rows.tgt, 4 * (size_t)M) || !get((void **)&rows.mw, 4 * (size_t)M) ||
            (dw && !get((void **)&rows.wt, 4 * (size_t)M)))
            return fail(LEIDEN_ERR_OOM, "leiden_csr_from_edges: device allocation failed");
        rows.len = rowlen;
        IK(cudaMemsetAsync(cnt, 0, 8 * (size_t)(n + 1), s));  // the cursors
        k_scatter_rows<<<grid_for(m, 256), 256, 0, s>>>(m, dsrc, ddst, dw, drop_self, rowstart, cnt, rows.tgt, rows.wt);
        IK(cudaGetLastError());
        if ((st = bins(rows, n, rowstart)) != LEIDEN_OK) return st;
        // ---- every row sorted and merged at the front of its segment
        int32_t ones = 1;  // the bits that targets have
        while (ones < n - 1) ones = 2 * ones + 1;
        IK(sort_segments(rows, (int64_t)hlongest, ones, combine, s));
        nlong = rows.count(6);
    }
    int64_t nover = nlong;
    const int32_t *llong = rows.list + rows.hb[6];
    int rbits = kRangeBits;
    if (nlong > 0) {  // (parts are numbered in 32 bits)
        while (((n - 1) >> rbits) + 1 > INT32_MAX / nlong) ++rbits;
        nrange = ((n - 1) >> rbits) + 1;
    }
    if (nrange > 1) {
        // ---- long rows: their entries by ranges of targets, each part as a row
        nparts = nlong * nrange;
        const int nr = (int)nrange;
        unsigned long long *pcnt = nullptr;
        int64_t *pstart = nullptr, entries = 0;
        void *ptmp = nullptr;
        if (!get((void **)&pcnt, 8 * (size_t)(nparts + 1)) || !get((void **)&pstart, 8 * (size_t)(nparts + 1)) ||
            !get((void **)&parts.len, 8 * (size_t)(nparts + 1)) || !get((void **)&so, 8 * (size_t)(nparts + 1)) ||
            !get((void **)&place, 8 * (size_t)nparts) || !get(&ptmp, scan_tmp_bytes(nparts + 1)))
            return fail(LEIDEN_ERR_OOM, "leiden_csr_from_edges: device allocation failed");
        const dim3 grid((unsigned)nlong, kBigSplit);
        IK(cudaMemsetAsync(pcnt, 0, 8 * (size_t)(nparts + 1), s));
        IK(cudaMemsetAsync(parts.len, 0, 8 * (size_t)(nparts + 1), s));
        k_split_rows<float, false><<<grid, 256, split_smem(nr, false), s>>>(llong, rowstart, nullptr, rows.tgt, nullptr,
                                                                            rbits, nr, pcnt, nullptr, nullptr, nullptr);
        IK(cudaGetLastError());
        IK(launch_exclusive_scan(reinterpret_cast<const int64_t *>(pcnt), pstart, nparts, ptmp, s));
        IK(cudaMemcpyAsync(&entries, pstart + nparts, 8, cudaMemcpyDeviceToHost, s));
        IK(cudaStreamSynchronize(s));
        if (!get((void **)&parts.tgt, 4 * (size_t)entries) || !get((void **)&parts.mw, 4 * (size_t)entries) ||
            (dw && !get((void **)&parts.wt, 4 * (size_t)entries)))
            return fail(LEIDEN_ERR_OOM, "leiden_csr_from_edges: device allocation failed");
        IK(cudaMemsetAsync(pcnt, 0, 8 * (size_t)(nparts + 1), s));
        k_split_rows<float, true><<<grid, 256, split_smem(nr, true), s>>>(llong, rowstart, nullptr, rows.tgt, rows.wt,
                                                                          rbits, nr, pcnt, pstart, parts.tgt, parts.wt);
        IK(cudaGetLastError());
        if ((st = bins(parts, nparts, pstart)) != LEIDEN_OK) return st;
        lmask = (int32_t)(((int64_t)1 << rbits) - 1);
        IK(sort_segments(parts, (int64_t)hlongest, lmask, combine, s));
        lg = &parts;
        nwords = ((int64_t)1 << rbits) / 32;
        nover = parts.count(6);
        lplace = place;
    }
    const int32_t *lover = lg->list + lg->hb[6];
    if (nover > 0) {
        // their merged lengths, from their bitmaps (kept for the output when
        // they all fit at once)
        at_once = std::max<int64_t>(1, std::min<int64_t>(nover, kBitmapBytes / (8 * nwords)));
        if (!get((void **)&bits, 8 * (size_t)(at_once * nwords)) || !get((void **)&abase, 8 * (size_t)(at_once + 1)))
            return fail(LEIDEN_ERR_OOM, "leiden_csr_from_edges: device allocation failed");
        before = bits + at_once * nwords;
    }
    auto map_long = [&](int64_t p0, int64_t c) -> cudaError_t {
        cudaError_t x = cudaMemsetAsync(bits, 0, 4 * (size_t)(c * nwords), s);
        if (x != cudaSuccess) return x;
        k_long_set<<<dim3((unsigned)c, kBigSplit), 256, 0, s>>>(lover, p0, lg->start, lg->tgt, lmask, bits, nwords);
        k_long_count<<<(unsigned)c, 1024, 0, s>>>(lover, p0, bits, before, nwords, lg->len);
        return cudaGetLastError();
    };
    for (int64_t p0 = 0; p0 < nover; p0 += at_once) IK(map_long(p0, std::min<int64_t>(at_once, nover - p0)));
    if (nparts > 0) {  // the long rows' lengths from their parts'
        void *ptmp = nullptr;
        if (!get(&ptmp, scan_tmp_bytes(nparts + 1)))
            return fail(LEIDEN_ERR_OOM, "leiden_csr_from_edges: device allocation failed");
        IK(launch_exclusive_scan(parts.len, so, nparts, ptmp, s));
        k_part_rows<<<grid_for(nlong, 256), 256, 0, s>>>(llong, nlong, (int)nrange, so, rowlen);
        IK(cudaGetLastError());
    }
    // ---- offsets: scan of the merged row lengths
    IK(launch_exclusive_scan(rowlen, doff, n, scan_tmp, s));
    IK(cudaMemcpyAsync(&nnz, doff + n, 8, cudaMemcpyDeviceToHost, s));
    IK(cudaStreamSynchronize(s));
    *nnz_io = nnz;
    if (nnz > cap || (nnz > 0 && (!indices || !weights)))
        return fail(LEIDEN_ERR_INVALID, "leiden_csr_from_edges: output capacity below the entry count");
    if (nnz > 0) {
        if (where == LEIDEN_HOST && (!get((void **)&sti, 4 * (size_t)nnz) || !get((void **)&stw, 4 * (size_t)nnz)))
            return fail(LEIDEN_ERR_OOM, "leiden_csr_from_edges: device allocation failed");
        IK(copy_segments(rows, doff, sti, stw, s));
        if (nparts > 0) {
            k_part_places<<<grid_for(nparts, 256), 256, 0, s>>>(llong, nparts, (int)nrange, so, doff, place);
            IK(cudaGetLastError());
            IK(copy_segments(parts, place, sti, stw, s));
        }
        int64_t *lens = nullptr;
        void *ltmp = nullptr;
        if (nover > 0 && (!get((void **)&lens, 8 * (size_t)at_once) || !get(&ltmp, scan_tmp_bytes(at_once + 1))))
            return fail(LEIDEN_ERR_OOM, "leiden_csr_from_edges: device allocation failed");
        for (int64_t p0 = 0; p0 < nover; p0 += at_once) {
            const int64_t c = std::min<int64_t>(at_once, nover - p0);
            if (nover > at_once) IK(map_long(p0, c));
            // where each one's sums start
            int64_t sums = 0;
            k_long_lens<<<grid_for(c, 256), 256, 0, s>>>(lover, p0, c, lg->len, lens);
            IK(cudaGetLastError());
            IK(launch_exclusive_scan(lens, abase, c, ltmp, s));
            IK(cudaMemcpyAsync(&sums, abase + c, 8, cudaMemcpyDeviceToHost, s));
            IK(cudaStreamSynchronize(s));
            double *acc = nullptr;
            if (cudaMallocAsync((void **)&acc, 8 * (size_t)(sums > 0 ? sums : 1), s) != cudaSuccess)
                return fail(LEIDEN_ERR_OOM, "leiden_csr_from_edges: device allocation failed");
            cudaMemsetAsync(acc, 0, 8 * (size_t)sums, s);
            const dim3 grid((unsigned)c, kBigSplit);
            k_long_place<<<grid, 256, 0, s>>>(lover, p0, lg->start, lg->tgt, lg->wt, combine, lmask, bits, before, nwords,
                                              lplace, sti, acc, abase);
            k_long_weights<<<grid, 256, 0, s>>>(lover, p0, lplace, lg->len, acc, abase, stw);
            e = cudaGetLastError();
            cudaFreeAsync(acc, s);
            IK(e);
        }
        if (where == LEIDEN_HOST) {
            IK(cudaMemcpyAsync(indices, sti, 4 * (size_t)nnz, out_kind, s));
            IK(cudaMemcpyAsync(weights, stw, 4 * (size_t)nnz, out_kind, s));
        }
    }
    IK(cudaMemcpyAsync(offsets, doff, 8 * (size_t)(n + 1), out_kind, s));
    IK(cudaStreamSynchronize(s));
#undef IK
    release();
    return LEIDEN_OK;
}

}  // namespace lgb
