// Rows of a holey CSR sorted by target: the deterministic mode writes every
// aggregated row in ascending target order (reading R10), so the stored
// super-vertex graph is the same bit for bit whatever order the hash tables
// held. The targets of a row differ from one another, so an entry's place is
// the number of smaller targets in its row, and each row is sorted by itself
// where it lies: communities of up to 32 member entries when the tile kernels
// of the aggregation write them; rows of up to 256 entries by a warp that
// counts smaller targets; of up to kRowSmem entries by a block in shared
// memory; longer ones are split by ranges of 2^kRangeBits targets
// (row_split.cuh), and each part goes back to its place in the row in order, by
// counting smaller targets or, from kPartCount entries, through a bitmap of its
// range in shared memory, whose running population count is every target's
// place. (Sorting all slots, unused ones included, as one sequence of (row,
// target) keys by 8-bit digits read and wrote some 50 bytes a slot and digit,
// four to seven digits: 45 of the 103 ms of a deterministic run of road
// 5000 x 5000.)
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "kernels.h"
#include "row_split.cuh"

namespace lgb {
namespace {

constexpr int kRowWarp = 256;    // longest row of a warp: eight entries a lane
constexpr int kRowSmem = 8192;   // longest row of a block: 16 bytes an entry of shared memory
constexpr int kBigSplit = 32;    // blocks that share a longer row
constexpr int kRangeBits = 18;   // bitmap and counts of a range: 64 KB of shared memory
constexpr int kPartCount = 1024; // longest part whose places are counted

// A warp per row of up to kRowWarp entries: its targets in shared memory, each
// lane counting the smaller ones of its up to eight, four targets a read.
__global__ void __launch_bounds__(256) k_sort_warp(const int32_t *__restrict__ list, int64_t count,
                                                   const int64_t *__restrict__ off, const int32_t *__restrict__ deg,
                                                   int32_t *idx, WInt *w) {
    __shared__ __align__(16) int32_t s_key[8][kRowWarp];
    const int lane = threadIdx.x & 31;
    int32_t *key = s_key[threadIdx.x >> 5];
    const int64_t warps = (int64_t)gridDim.x * 8;
    for (int64_t t = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); t < count; t += warps) {
        const int32_t c = list[t];
        const int32_t d = deg[c];
        if (d <= 1 || d > kRowWarp) continue;  // bins bound d: longer rows never come here
        const int64_t o = off[c];
        const int pad = (d + 3) & ~3;
        int32_t k[8], rank[8];
        WInt x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int e = q * 32 + lane;
            k[q] = INT32_MAX;
            x[q] = 0;
            rank[q] = 0;
            if (e < d) {
                k[q] = idx[o + e];
                x[q] = w[o + e];
            }
            if (e < pad) key[e] = k[q];
        }
        __syncwarp();
        const int n = (d + 31) / 32;  // entries of a lane
        for (int e = 0; e < pad; e += 4) {
            const int4 y = *reinterpret_cast<const int4 *>(&key[e]);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q < n) rank[q] += (y.x < k[q]) + (y.y < k[q]) + (y.z < k[q]) + (y.w < k[q]);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (q * 32 + lane < d) {
                idx[o + rank[q]] = k[q];
                w[o + rank[q]] = x[q];
            }
        __syncwarp();
    }
}

// A block per row of up to kRowSmem entries: (target, place) words sorted by
// a bitonic network in shared memory, then the weights follow their places.
__global__ void k_sort_block(const int32_t *__restrict__ list, int64_t count, const int64_t *__restrict__ off,
                             const int32_t *__restrict__ deg, int32_t *idx, WInt *w, int cap) {
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned long long *key = reinterpret_cast<unsigned long long *>(smem);
    WInt *x = reinterpret_cast<WInt *>(smem) + cap;
    for (int64_t t = blockIdx.x; t < count; t += gridDim.x) {
        const int32_t c = list[t];
        const int32_t d = deg[c];
        if (d <= 1 || d > cap) continue;  // the same in every thread
        const int64_t o = off[c];
        int P = 32;
        while (P < d) P <<= 1;
        for (int e = threadIdx.x; e < P; e += blockDim.x) {
            key[e] = e < d ? ((unsigned long long)(uint32_t)idx[o + e] << 32) | (uint32_t)e : ~0ULL;
            if (e < d) x[e] = w[o + e];
        }
        __syncthreads();
        for (int size = 2; size <= P; size <<= 1)
            for (int st = size >> 1; st > 0; st >>= 1) {
                for (int i = threadIdx.x; i < P / 2; i += blockDim.x) {
                    const int lo = 2 * i - (i & (st - 1));
                    const unsigned long long p = key[lo], q = key[lo + st];
                    if ((p > q) == ((lo & size) == 0)) {
                        key[lo] = q;
                        key[lo + st] = p;
                    }
                }
                __syncthreads();
            }
        for (int e = threadIdx.x; e < d; e += blockDim.x) {
            const unsigned long long k = key[e];
            idx[o + e] = (int32_t)(k >> 32);
            w[o + e] = x[(uint32_t)k];
        }
        __syncthreads();
    }
}

// ---- rows of more than kRowSmem entries
__global__ void k_big_rows(const int32_t *list, int64_t count, const int32_t *deg, int32_t *big, unsigned *nbig) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < count; t += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = list[t];
        if (deg[c] > kRowSmem) big[atomicAdd(nbig, 1u)] = c;
    }
}
// a block per part: part k of row big[k / nr] has the entries [start[k],
// start[k + 1]) of (cidx, cw), whose targets differ and agree above kRangeBits
constexpr int kRangeWords = (1 << kRangeBits) / 32;
__global__ void __launch_bounds__(512) k_sort_parts(const int32_t *__restrict__ big, int64_t nparts, int nr,
                                                    const int64_t *__restrict__ start,
                                                    const int64_t *__restrict__ off, const int32_t *__restrict__ cidx,
                                                    const WInt *__restrict__ cw, int32_t *idx, WInt *w) {
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned *bits = reinterpret_cast<unsigned *>(smem);            // [kRangeWords]
    unsigned *before = bits + kRangeWords;                          // targets before each word
    int32_t *key = reinterpret_cast<int32_t *>(smem);               // [kPartCount], over the bitmap
    __shared__ unsigned s_part[16];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    constexpr int per = kRangeWords / 512;  // words of a thread
    for (int64_t k = blockIdx.x; k < nparts; k += gridDim.x) {
        const int64_t b = start[k], c = start[k + 1] - b, p = k / nr;
        if (c == 0) continue;  // the same in every thread
        const int64_t o = off[big[p]] + (b - start[p * nr]);
        if (c <= kPartCount) {
            const int pad = ((int)c + 3) & ~3;
            for (int e = threadIdx.x; e < pad; e += blockDim.x) key[e] = e < c ? cidx[b + e] : INT32_MAX;
            __syncthreads();
            for (int e = threadIdx.x; e < c; e += blockDim.x) {
                const int32_t x = key[e];
                int rank = 0;
                for (int j = 0; j < pad; j += 4) {
                    const int4 y = *reinterpret_cast<const int4 *>(&key[j]);
                    rank += (y.x < x) + (y.y < x) + (y.z < x) + (y.w < x);
                }
                idx[o + rank] = x;
                w[o + rank] = cw[b + e];
            }
        } else {
            for (int q = threadIdx.x; q < kRangeWords; q += blockDim.x) bits[q] = 0u;
            __syncthreads();
            for (int64_t e = threadIdx.x; e < c; e += blockDim.x) {
                const int32_t x = cidx[b + e] & ((1 << kRangeBits) - 1);
                atomicOr(&bits[x >> 5], 1u << (x & 31));
            }
            __syncthreads();
            // running population count: warp by warp of consecutive words
            unsigned run = 0;
            for (int q = 0; q < per; ++q) {
                const int at = (wib * per + q) * 32 + lane;
                const unsigned own = __popc(bits[at]);
                unsigned inc = own;
                for (int s = 1; s < 32; s <<= 1) {
                    const unsigned y = __shfl_up_sync(kFull, inc, s);
                    if (lane >= s) inc += y;
                }
                before[at] = run + inc - own;
                run += __shfl_sync(kFull, inc, 31);
            }
            if (lane == 0) s_part[wib] = run;
            __syncthreads();
            for (int64_t e = threadIdx.x; e < c; e += blockDim.x) {
                const int32_t x = cidx[b + e], at = (x & ((1 << kRangeBits) - 1)) >> 5;
                int64_t pos = o + before[at] + __popc(bits[at] & ((1u << (x & 31)) - 1u));
                for (int q = 0; q < at / (32 * per); ++q) pos += s_part[q];  // the words of the warps before
                idx[pos] = x;
                w[pos] = cw[b + e];
            }
        }
        __syncthreads();
    }
}

inline int blocks_for(int64_t items, int64_t most) { return (int)std::max<int64_t>(1, std::min(items, most)); }

}  // namespace

cudaError_t launch_sort_rows(int bin, const int32_t *list, int64_t count, int64_t n, const int64_t *off,
                             const int32_t *deg, int32_t *idx, WInt *w, int64_t max_row, int sms, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    cudaError_t e;
    if (bin <= 4) {
        k_sort_warp<<<blocks_for((count + 7) / 8, (int64_t)sms * 8), 256, 0, s>>>(list, count, off, deg, idx, w);
        return cudaGetLastError();
    }
    // rows of bin 5 have up to kBlockMaxDeg entries; bin 6 takes all the
    // shared memory a row may need, bounded by the longest row's capacity
    int cap = kBlockMaxDeg;
    if (bin > 5)
        while (cap < max_row && cap < kRowSmem) cap <<= 1;
    const size_t bytes = (size_t)cap * 16;
    if ((e = cudaFuncSetAttribute(k_sort_block, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmem * 16)) !=
        cudaSuccess)
        return e;
    k_sort_block<<<blocks_for(count, (int64_t)sms * 8), cap > kBlockMaxDeg ? 512 : 256, bytes, s>>>(list, count, off, deg,
                                                                                               idx, w, cap);
    if ((e = cudaGetLastError()) != cudaSuccess || bin <= 5 || max_row <= kRowSmem) return e;
    // longer rows
    int32_t *big = nullptr, *cidx = nullptr;
    WInt *cw = nullptr;
    int64_t *start = nullptr;
    unsigned long long *cnt = nullptr;
    unsigned *nbig = nullptr;
    unsigned nb = 0;
    void *stmp = nullptr;
    auto get = [&](auto **p, size_t bytes2) {
        return cudaMallocAsync(reinterpret_cast<void **>(p), bytes2, s);
    };
    auto done = [&](cudaError_t r) {
        for (void *p : {(void *)big, (void *)cidx, (void *)cw, (void *)start, (void *)cnt, (void *)nbig, stmp})
            if (p) cudaFreeAsync(p, s);
        return r;
    };
    if ((e = get(&big, 4 * (size_t)count)) != cudaSuccess || (e = get(&nbig, sizeof(unsigned))) != cudaSuccess)
        return done(e);
    if ((e = cudaMemsetAsync(nbig, 0, sizeof(unsigned), s)) != cudaSuccess) return done(e);
    k_big_rows<<<blocks_for((count + 255) / 256, (int64_t)sms * 8), 256, 0, s>>>(list, count, deg, big, nbig);
    if ((e = cudaGetLastError()) != cudaSuccess ||
        (e = cudaMemcpyAsync(&nb, nbig, sizeof(nb), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaStreamSynchronize(s)) != cudaSuccess || nb == 0)
        return done(e);
    // their entries by ranges of targets, then every part back to its place
    const int nr = (int)(((n - 1) >> kRangeBits) + 1);
    const int64_t nparts = (int64_t)nb * nr;
    int64_t entries = 0;
    if ((e = get(&cnt, 8 * (size_t)(nparts + 1))) != cudaSuccess ||
        (e = get(&start, 8 * (size_t)(nparts + 1))) != cudaSuccess ||
        (e = get(&stmp, scan_tmp_bytes(nparts + 1))) != cudaSuccess ||
        (e = cudaMemsetAsync(cnt, 0, 8 * (size_t)(nparts + 1), s)) != cudaSuccess)
        return done(e);
    const dim3 grid(nb, kBigSplit);
    const size_t smem = split_smem(nr, true);
    if ((e = cudaFuncSetAttribute(k_split_rows<WInt, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)smem)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(k_sort_parts, cudaFuncAttributeMaxDynamicSharedMemorySize, 8 * kRangeWords)) !=
            cudaSuccess)
        return done(e);
    k_split_rows<WInt, false><<<grid, 256, split_smem(nr, false), s>>>(big, off, deg, idx, nullptr, kRangeBits, nr, cnt,
                                                                       nullptr, nullptr, nullptr);
    if ((e = cudaGetLastError()) != cudaSuccess ||
        (e = launch_exclusive_scan(reinterpret_cast<const int64_t *>(cnt), start, nparts, stmp, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(&entries, start + nparts, 8, cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaStreamSynchronize(s)) != cudaSuccess ||
        (e = get(&cidx, 4 * (size_t)entries)) != cudaSuccess || (e = get(&cw, 8 * (size_t)entries)) != cudaSuccess ||
        (e = cudaMemsetAsync(cnt, 0, 8 * (size_t)(nparts + 1), s)) != cudaSuccess)
        return done(e);
    k_split_rows<WInt, true><<<grid, 256, smem, s>>>(big, off, deg, idx, w, kRangeBits, nr, cnt, start, cidx, cw);
    k_sort_parts<<<blocks_for(nparts, (int64_t)sms * 3), 512, 8 * kRangeWords, s>>>(big, nparts, nr, start, off, cidx,
                                                                                   cw, idx, w);
    return done(cudaGetLastError());
}

}  // namespace lgb
