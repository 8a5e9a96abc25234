// Rows of a holey CSR sorted by target: the deterministic mode writes every
// aggregated row in ascending target order (reading R10), so the stored
// super-vertex graph is the same bit for bit whatever order the hash tables
// held. The targets of a row differ from one another, so an entry's place is
// the number of smaller targets in its row, and each row is sorted by itself
// where it lies: communities of up to 32 member entries when the tile kernels
// of the aggregation write them; rows of up to 256 entries by a warp that
// counts smaller targets; of up to kRowSmem entries by a block in shared
// memory; longer ones through a bitmap of their targets, whose running
// population count is every target's place. (Sorting all slots, unused ones
// included, as one sequence of (row, target) keys by 8-bit digits read and
// wrote some 50 bytes a slot and digit, four to seven digits: 45 of the 103 ms
// of a deterministic run of road 5000 x 5000.)
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace lgb {
namespace {

constexpr int kRowWarp = 256;    // longest row of a warp: eight entries a lane
constexpr int kRowSmem = 8192;   // longest row of a block: 16 bytes an entry of shared memory
constexpr int kBigSplit = 32;    // blocks that share a longer row
constexpr int64_t kBitmapBytes = (int64_t)1 << 30;  // bitmaps and their counts, for the rows taken at once

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
__global__ void k_big_rows(const int32_t *list, int64_t count, const int32_t *deg, int32_t *big, int32_t *bdeg,
                           unsigned *nbig) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < count; t += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = list[t];
        if (deg[c] <= kRowSmem) continue;
        const unsigned p = atomicAdd(nbig, 1u);
        big[p] = c;
        bdeg[p] = deg[c];
    }
}
// row blockIdx.x of the rows taken at once: its entries to the scratch, its
// targets into its bitmap
__global__ void k_big_set(const int32_t *big, const int64_t *boff, int64_t p0, const int64_t *off, const int32_t *idx,
                          const WInt *w, int32_t *cidx, WInt *cw, unsigned *bits, int64_t nwords) {
    const int64_t p = p0 + blockIdx.x, o = off[big[p]], b = boff[p], d = boff[p + 1] - b;
    unsigned *m = bits + (int64_t)blockIdx.x * nwords;
    for (int64_t e = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; e < d; e += (int64_t)gridDim.y * blockDim.x) {
        const int32_t k = idx[o + e];
        cidx[b + e] = k;
        cw[b + e] = w[o + e];
        atomicOr(&m[k >> 5], 1u << (k & 31));
    }
}
// targets of row blockIdx.x before each word of its bitmap
__global__ void __launch_bounds__(1024) k_big_count(const unsigned *bits, unsigned *before, int64_t nwords) {
    __shared__ unsigned s_w[32];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const unsigned *m = bits + (int64_t)blockIdx.x * nwords;
    unsigned *out = before + (int64_t)blockIdx.x * nwords;
    unsigned carry = 0;
    for (int64_t i0 = 0; i0 < nwords; i0 += blockDim.x) {
        const int64_t i = i0 + threadIdx.x;
        const unsigned own = i < nwords ? __popc(m[i]) : 0;
        unsigned inc = own;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) s_w[wib] = inc;
        __syncthreads();
        unsigned mine = carry, all = 0;
        for (int k = 0; k < 32; ++k) {
            if (k < wib) mine += s_w[k];
            all += s_w[k];
        }
        if (i < nwords) out[i] = mine + inc - own;
        carry += all;
        __syncthreads();
    }
}
__global__ void k_big_place(const int32_t *big, const int64_t *boff, int64_t p0, const int64_t *off,
                            const int32_t *cidx, const WInt *cw, const unsigned *bits, const unsigned *before,
                            int64_t nwords, int32_t *idx, WInt *w) {
    const int64_t p = p0 + blockIdx.x, o = off[big[p]], b = boff[p], d = boff[p + 1] - b;
    const unsigned *m = bits + (int64_t)blockIdx.x * nwords, *f = before + (int64_t)blockIdx.x * nwords;
    for (int64_t e = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; e < d; e += (int64_t)gridDim.y * blockDim.x) {
        const int32_t k = cidx[b + e];
        const int64_t at = o + f[k >> 5] + __popc(m[k >> 5] & ((1u << (k & 31)) - 1u));
        idx[at] = k;
        w[at] = cw[b + e];
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
    int64_t *boff = nullptr;
    unsigned *nbig = nullptr, *bits = nullptr;
    unsigned nb = 0;
    void *stmp = nullptr;
    auto get = [&](auto **p, size_t bytes2) {
        return cudaMallocAsync(reinterpret_cast<void **>(p), bytes2, s);
    };
    auto done = [&](cudaError_t r) {
        for (void *p : {(void *)big, (void *)cidx, (void *)cw, (void *)boff, (void *)nbig, (void *)bits, stmp})
            if (p) cudaFreeAsync(p, s);
        return r;
    };
    if ((e = get(&big, 8 * (size_t)count)) != cudaSuccess || (e = get(&nbig, sizeof(unsigned))) != cudaSuccess)
        return done(e);
    int32_t *bdeg = big + count;
    if ((e = cudaMemsetAsync(nbig, 0, sizeof(unsigned), s)) != cudaSuccess) return done(e);
    k_big_rows<<<blocks_for((count + 255) / 256, (int64_t)sms * 8), 256, 0, s>>>(list, count, deg, big, bdeg, nbig);
    if ((e = cudaGetLastError()) != cudaSuccess ||
        (e = cudaMemcpyAsync(&nb, nbig, sizeof(nb), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaStreamSynchronize(s)) != cudaSuccess || nb == 0)
        return done(e);
    int64_t entries = 0;
    if ((e = get(&boff, 8 * ((size_t)nb + 1))) != cudaSuccess || (e = get(&stmp, scan_tmp_bytes(nb))) != cudaSuccess ||
        (e = launch_exclusive_scan_i32(bdeg, boff, nb, stmp, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(&entries, boff + nb, 8, cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaStreamSynchronize(s)) != cudaSuccess)
        return done(e);
    const int64_t nwords = (n + 31) / 32;
    const int64_t rows = std::max<int64_t>(1, std::min<int64_t>(nb, kBitmapBytes / (8 * nwords)));
    if ((e = get(&cidx, 4 * (size_t)entries)) != cudaSuccess || (e = get(&cw, 8 * (size_t)entries)) != cudaSuccess ||
        (e = get(&bits, 8 * (size_t)(rows * nwords))) != cudaSuccess)
        return done(e);
    unsigned *before = bits + rows * nwords;
    for (int64_t p0 = 0; p0 < (int64_t)nb; p0 += rows) {
        const int64_t r = std::min<int64_t>(rows, (int64_t)nb - p0);
        const dim3 grid((unsigned)r, kBigSplit);
        if ((e = cudaMemsetAsync(bits, 0, 4 * (size_t)(r * nwords), s)) != cudaSuccess) return done(e);
        k_big_set<<<grid, 256, 0, s>>>(big, boff, p0, off, idx, w, cidx, cw, bits, nwords);
        k_big_count<<<(unsigned)r, 1024, 0, s>>>(bits, before, nwords);
        k_big_place<<<grid, 256, 0, s>>>(big, boff, p0, off, cidx, cw, bits, before, nwords, idx, w);
        if ((e = cudaGetLastError()) != cudaSuccess) return done(e);
    }
    return done(cudaSuccess);
}

}  // namespace lgb
