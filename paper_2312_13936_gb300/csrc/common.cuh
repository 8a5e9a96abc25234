// Device-side building blocks shared by the Leiden kernels (sm_103a).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace lgb {

constexpr int kWarp = 32;
constexpr unsigned kFull = 0xffffffffu;

// Arithmetic policies. acc is the type of vertex weights K_i; sum that of
// per-edge sums K_{i->c}; key the type of move keys and their gains; tot the
// type of community totals Sigma_c and of the asynchronous sweep's
// delta-modularity sums. The deterministic mode decides moves in exact
// integer arithmetic on integer weights: sums, K and Sigma in int64, keys
// (products of two such sums) in 128 bits, and a sweep's gain sum in 128
// bits (two 64-bit words, lo then hi). Det64 is the same arithmetic for
// graphs of 2m < 2^31, where it is exact in narrower words: every sum of
// entries is at most 2m and fits in 32 bits, every product is below 2^62 and
// every key and gain fits in 64; the decisions are the same bit for bit. (A
// 128-bit key took twice the registers of a 64-bit one and spilled at 64
// registers a thread, and shared memory has no 64-bit add: every insertion
// was a compare-and-swap loop.) The asynchronous mode keeps Sigma and 2m in
// fp64 and everything per edge in fp32: on this GPU the fp64 pipe is a small
// fraction of the fp32 rate, and the move key
// K_{i->c} - gamma K_i Sigma_c / 2m has terms of the order of K_i, so fp32
// keeps its relative precision. packed: a global table's slot is one 8-byte
// word of a key and a 32-bit sum.
struct Det {
    using acc = long long;
    using sum = long long;
    using tot = long long;
    using key = __int128;
    static constexpr bool det = true, packed = false;
};
struct Det64 {
    using acc = long long;
    using sum = int32_t;
    using tot = long long;
    using key = long long;
    static constexpr bool det = true, packed = true;
};
struct Async {
    using acc = float;
    using sum = float;
    using tot = double;
    using key = float;
    static constexpr bool det = false, packed = true;
};

template <class A> struct AccLimits;
template <> struct AccLimits<long long> {
    __device__ static constexpr long long lowest() { return (long long)0x8000000000000000ULL; }
};
template <> struct AccLimits<double> {
    __device__ static double lowest() { return __longlong_as_double(0xfff0000000000000LL); }  // -inf
};
template <> struct AccLimits<float> {
    __device__ static float lowest() { return __int_as_float(0xff800000); }  // -inf
};
template <> struct AccLimits<__int128> {
    __device__ static __int128 lowest() { return (__int128)((unsigned __int128)1 << 127); }
};

// Register shuffles of the key types (a 128-bit key moves as two words).
__device__ __forceinline__ float kshfl_xor(unsigned mask, float x, int o, int w = 32) {
    return __shfl_xor_sync(mask, x, o, w);
}
__device__ __forceinline__ long long kshfl_xor(unsigned mask, long long x, int o, int w = 32) {
    return __shfl_xor_sync(mask, x, o, w);
}
__device__ __forceinline__ __int128 kshfl_xor(unsigned mask, __int128 x, int o, int w = 32) {
    const unsigned long long lo = __shfl_xor_sync(mask, (unsigned long long)x, o, w);
    const long long hi = __shfl_xor_sync(mask, (long long)(x >> 64), o, w);
    return (__int128)(((unsigned __int128)(unsigned long long)hi << 64) | lo);
}
// A 128-bit unsigned sum held as two words (lo, hi) in global memory:
// atomically add x, carrying into hi when lo wraps. Every addition that
// wraps lo adds exactly one carry, so the pair is the exact sum mod 2^128
// in any order.
__device__ __forceinline__ void atomic_add_u128(unsigned long long *p, unsigned __int128 x) {
    const unsigned long long lo = (unsigned long long)x;
    unsigned long long hi = (unsigned long long)(x >> 64);
    if (lo) {
        const unsigned long long old = atomicAdd(&p[0], lo);
        if (old + lo < old) hi += 1ULL;
    }
    if (hi) atomicAdd(&p[1], hi);
}


template <class A, class W> __device__ __forceinline__ A wconv(W w) { return (A)w; }

__device__ __forceinline__ void atomic_add_acc(long long *p, long long v) {
    atomicAdd(reinterpret_cast<unsigned long long *>(p), static_cast<unsigned long long>(v));
}
__device__ __forceinline__ void atomic_add_acc(double *p, double v) { atomicAdd(p, v); }
__device__ __forceinline__ void atomic_add_acc(float *p, float v) { atomicAdd(p, v); }
__device__ __forceinline__ void atomic_add_acc(unsigned long long *p, unsigned long long v) { atomicAdd(p, v); }
__device__ __forceinline__ void atomic_add_acc(int32_t *p, int32_t v) { atomicAdd(p, v); }

// Running per-graph sum of one thread (sweep gains, move counts). In a batch
// of graphs the sum of the previous graph goes to its slot base[g] when the
// thread reaches a vertex of another graph; a single graph never flushes
// here and reduces per warp at the end of the sweep instead.
template <class V> struct GAcc {
    V v = 0;
    int32_t g = 0;
};
template <class V, class D>
__device__ __forceinline__ void gacc_add(GAcc<V> &acc, bool batch, int32_t g, V x, D *base) {
    if (batch && g != acc.g) {
        if (acc.v != (V)0) atomic_add_acc(&base[acc.g], (D)acc.v);
        acc.v = 0;
        acc.g = g;
    }
    acc.v += x;
}
template <class V, class D> __device__ __forceinline__ void gacc_flush(GAcc<V> &acc, D *base) {
    if (acc.v != (V)0) atomic_add_acc(&base[acc.g], (D)acc.v);
    acc.v = 0;
}

// The deterministic mode's gain sums: 128 bits per thread, flushed into
// per-graph slots of two words (lo, hi) at base + 2 g.
__device__ __forceinline__ void gacc_add(GAcc<unsigned __int128> &acc, bool batch, int32_t g, unsigned __int128 x,
                                         unsigned long long *base) {
    if (batch && g != acc.g) {
        if (acc.v) atomic_add_u128(base + 2 * (size_t)acc.g, acc.v);
        acc.v = 0;
        acc.g = g;
    }
    acc.v += x;
}
__device__ __forceinline__ void gacc_flush(GAcc<unsigned __int128> &acc, unsigned long long *base) {
    if (acc.v) atomic_add_u128(base + 2 * (size_t)acc.g, acc.v);
    acc.v = 0;
}
__device__ __forceinline__ unsigned __int128 warp_sum_u128(unsigned __int128 v) {
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)v, o);
        const unsigned long long hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)(v >> 64), o);
        v += ((unsigned __int128)hi << 64) | lo;
    }
    return v;
}

// Σ reads: the async mode sees concurrent atomics from other SMs, so it reads
// through L2 (ld.global.cg); deterministic mode reads a snapshot.
template <class A> __device__ __forceinline__ A load_cg(const A *p) { return __ldcg(p); }

// Move keys (Eq. 2). Deterministic mode, Eq. 2 times 2m^2 (kscale = 2m), in
// 128 bits (each product is below (2m)^2; Det64: 64 bits):
//   key(c) = 2m K_{i->c} - K_i Sigma_c,  stay = 2m K_{i->d} - K_i (Sigma_d - K_i).
// Asynchronous mode, Eq. 2 times m (kscale = 1/2m):
//   key(c) = K_{i->c} - gamma K_i Sigma_c / 2m,  stay = K_{i->d} - gamma K_i (Sigma_d - K_i) / 2m.
// The vertex moves to c* iff key(c*) > stay; the gain key(c*) - stay is
// 2m^2 dQ (deterministic) or m dQ (asynchronous).
__device__ __forceinline__ __int128 move_key(long long two_m, long long kic, long long ki, long long sc, double) {
    return (__int128)two_m * kic - (__int128)ki * sc;
}
__device__ __forceinline__ long long move_key(long long two_m, int32_t kic, long long ki, long long sc, double) {
    return two_m * kic - ki * sc;  // Det64
}
__device__ __forceinline__ float move_key(float inv2m, float kic, float ki, double sc, double gamma) {
    return kic - (float)gamma * ki * ((float)sc * inv2m);
}
__device__ __forceinline__ __int128 stay_key(long long two_m, long long kid, long long ki, long long sd, double) {
    return (__int128)two_m * kid - (__int128)ki * (sd - ki);
}
__device__ __forceinline__ long long stay_key(long long two_m, int32_t kid, long long ki, long long sd, double) {
    return two_m * kid - ki * (sd - ki);  // Det64
}
__device__ __forceinline__ float stay_key(float inv2m, float kid, float ki, double sd, double gamma) {
    return kid - (float)gamma * ki * (((float)sd - ki) * inv2m);
}

// SplitMix64 (Steele, Lea & Flood, OOPSLA 2014): output number i+1 of the
// generator whose state starts at s. Vertex priorities of the sweep schedule.
__device__ __forceinline__ uint64_t splitmix64_at(uint64_t s, uint64_t i) {
    uint64_t z = s + (i + 1ULL) * 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}
// u precedes v in the schedule order: higher priority first, ties by id.
__device__ __forceinline__ bool precedes(uint64_t pu, int32_t u, uint64_t pv, int32_t v) {
    return pu > pv || (pu == pv && u < v);
}

// Open-addressing hash table with linear probing (keys -1 = empty).
__device__ __forceinline__ uint32_t hslot(int32_t key, int bits) {
    return ((uint32_t)key * 0x9E3779B1u) >> (32 - bits);
}
// the slot of key k, taken for it if it has none yet (fresh); -1: no room
__device__ __forceinline__ int hash_slot(int32_t *keys, int bits, int32_t k, bool &fresh) {
    const uint32_t mask = (1u << bits) - 1u;
    uint32_t s = hslot(k, bits);
    for (uint32_t probe = 0; probe <= mask; ++probe) {
        int32_t cur = *((volatile int32_t *)&keys[s]);
        if (cur == -1) {
            cur = atomicCAS(&keys[s], -1, k);
            fresh = cur == -1;
            if (fresh) return (int)s;
        }
        if (cur == k) return (int)s;
        s = (s + 1u) & mask;
    }
    return -1;
}
// (The sum is added inside the probing loop: with hash_slot and the addition
// after it, as the rows that stay in registers need it, the persistent sweeps
// that insert with this spilled 2.5 KB at 64 registers a thread instead of
// nothing.)
template <class A>
__device__ __forceinline__ bool hash_add(int32_t *keys, A *vals, int bits, int32_t k, A v) {
    const uint32_t mask = (1u << bits) - 1u;
    uint32_t s = hslot(k, bits);
    for (uint32_t probe = 0; probe <= mask; ++probe) {
        int32_t cur = *((volatile int32_t *)&keys[s]);
        if (cur == k) {
            atomic_add_acc(&vals[s], v);
            return true;
        }
        if (cur == -1) {
            int32_t prev = atomicCAS(&keys[s], -1, k);
            if (prev == -1 || prev == k) {
                atomic_add_acc(&vals[s], v);
                return true;
            }
        }
        s = (s + 1u) & mask;
    }
    return false;
}

// Open-addressing table whose slot is one 8-byte word: the key in the low
// half (-1: empty), a 32-bit sum (fp32, or an integer of Det64) in the high
// half, so that an insertion touches one memory sector. A new key goes in
// with its value by one 64-bit compare-and-swap against the empty word; a
// failed swap returns the slot's word, and if its key is ours the value is
// added to the high half. A slot's key never changes once set, so the key
// half of a returned word is exact even while other threads add to its value
// half.
constexpr unsigned long long kEmptyKV = 0x00000000ffffffffULL;  // key -1, value 0 (0.0f)
__device__ __forceinline__ unsigned kv_bits(float v) { return __float_as_uint(v); }
__device__ __forceinline__ unsigned kv_bits(int32_t v) { return (unsigned)v; }
__device__ __forceinline__ void kv_value(unsigned long long w, float &v) { v = __uint_as_float((uint32_t)(w >> 32)); }
__device__ __forceinline__ void kv_value(unsigned long long w, int32_t &v) { v = (int32_t)(uint32_t)(w >> 32); }
template <class V> __device__ __forceinline__ bool hash_add_kv(unsigned long long *kv, int bits, int32_t k, V v) {
    const uint32_t mask = (1u << bits) - 1u;
    const unsigned long long mine = ((unsigned long long)kv_bits(v) << 32) | (uint32_t)k;
    uint32_t s = hslot(k, bits);
    for (uint32_t probe = 0; probe <= mask; ++probe) {
        const unsigned long long cur = atomicCAS(&kv[s], kEmptyKV, mine);
        if (cur == kEmptyKV) return true;
        if ((int32_t)(uint32_t)cur == k) {
            atomicAdd(reinterpret_cast<V *>(&kv[s]) + 1, v);
            return true;
        }
        s = (s + 1u) & mask;
    }
    return false;
}

__device__ __forceinline__ int ceil_log2(int64_t x) {
    int b = 0;
    while ((1LL << b) < x) ++b;
    return b;
}

template <class T> __device__ __forceinline__ T warp_sum(T v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// Row i of a CSR against labels C: K_i (sum of weights) and the weight to
// vertices labelled ci, over entries [from, to) of the row with stride step,
// four entries in flight.
__device__ __forceinline__ void row_part(const int32_t *__restrict__ idx, const float *__restrict__ w,
                                         const int32_t *__restrict__ C, int64_t e0, int64_t from, int64_t to, int step,
                                         int32_t ci, double &k, double &in) {
    for (int64_t e = e0 + from; e < e0 + to; e += 4 * (int64_t)step) {
        int32_t j[4], c[4];
        float x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bool has = e + q * step < e0 + to;
            j[q] = has ? idx[e + q * step] : -1;
            x[q] = !has ? 0.0f : w ? w[e + q * step] : 1.0f;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) c[q] = j[q] >= 0 ? C[j[q]] : -1;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (j[q] >= 0) {
                k += (double)x[q];
                if (c[q] == ci) in += (double)x[q];
            }
    }
}
// the same for every lane's row of a full warp: short rows by their lane,
// rows longer than 64 entries (LONG) by the whole warp in turn (valid: the
// lane has a row)
template <bool LONG>
__device__ __forceinline__ void warp_rows(const int64_t *off, const int32_t *idx, const float *w, const int32_t *C,
                                          bool valid, int64_t i, int32_t ci, double &k, double &in) {
    const int lane = threadIdx.x & 31;
    int64_t e0 = 0, d = 0;
    if (valid) {
        e0 = off[i];
        d = off[i + 1] - e0;
        if (!LONG || d <= 64) row_part(idx, w, C, e0, 0, d, 1, ci, k, in);
    }
    unsigned longs = LONG ? __ballot_sync(kFull, valid && d > 64) : 0u;
    while (longs) {
        const int src = __ffs(longs) - 1;
        longs &= longs - 1;
        double kl = 0, il = 0;
        row_part(idx, w, C, __shfl_sync(kFull, e0, src), lane, __shfl_sync(kFull, d, src), 32,
                 __shfl_sync(kFull, ci, src), kl, il);
        kl = warp_sum(kl);
        il = warp_sum(il);
        if (lane == src) {
            k = kl;
            in = il;
        }
    }
}

// arr[key] += x for every lane of a full warp (key < 0: nothing), with one
// atomic per distinct key: lanes that share a key sum first. Cheap when a
// warp's keys repeat (labels of nearby vertices).
__device__ __forceinline__ void warp_add_by_key(double *arr, int64_t key, double x) {
    unsigned todo = __ballot_sync(kFull, key >= 0);
    while (todo) {
        const int lead = __ffs(todo) - 1;
        const int64_t k = __shfl_sync(kFull, key, lead);
        const unsigned same = __ballot_sync(kFull, key == k);
        const double s = warp_sum(key == k ? x : 0.0);
        if ((int)(threadIdx.x & 31) == lead && s != 0.0) atomicAdd(&arr[k], s);
        todo &= ~same;
    }
}

// Sum over a full warp, in one instruction for 32-bit integers.
template <class T> __device__ __forceinline__ T full_sum(T v) { return warp_sum(v); }
__device__ __forceinline__ int32_t full_sum(int32_t v) { return __reduce_add_sync(kFull, v); }

// Sum of v over the lanes of peers (every lane of peers calls it, with the
// same peers).
template <class A>
__device__ __forceinline__ A peer_sum(unsigned peers, A v) {
    if (peers == kFull) return warp_sum(v);
    // alone: no shuffle (lanes of different peers run one group after another,
    // so 32 groups of one took 32 turns)
    if ((peers & (peers - 1u)) == 0u) return v;
    A s = 0;
    for (unsigned m = peers; m; m &= m - 1) s += __shfl_sync(peers, v, __ffs(m) - 1);
    return s;
}

// Profiling counters: every lane holds partial counts, flushed with one atomic
// per warp at the end. 32 bits hold a lane's share of a launch's rows of up to
// kWarpMaxDeg entries (64 took the two-block sweeps' spills from 0.5 to 0.7
// KB); the entries of longer rows, which one lane counts for its block or for
// the whole grid, are added in memory as they come (prof_add).
struct ProfCounts {
    unsigned v[6] = {0, 0, 0, 0, 0, 0};
    __device__ __forceinline__ void flush(unsigned long long *dst) {
        if (!dst) return;
        for (int k = 0; k < 6; ++k) {
            const unsigned long long s = warp_sum((unsigned long long)v[k]);
            if ((threadIdx.x & 31) == 0 && s) atomicAdd(&dst[k], s);
        }
    }
};
__device__ __forceinline__ void prof_add(unsigned long long *dst, int k, int64_t x) {
    if (dst) atomicAdd(&dst[k], (unsigned long long)x);
}

// Device error word: kernels record the first failure here instead of
// trapping; the host reads it after each phase.
enum : int { kErrNone = 0, kErrHashFull = 1, kErrBadIndex = 2, kErrTimeout = 3 };
__device__ __forceinline__ void set_error(int *err, int code) {
    if (err) atomicCAS(err, 0, code);
}

__device__ __forceinline__ unsigned bar_poll(const unsigned *p) {
    unsigned r;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(r) : "l"(p) : "memory");
    return r;
}
// Grid-wide barrier of a cooperative launch: one arrival counter, zero when
// the launch begins (the launcher clears it), that thread 0 of every block
// adds to (release, no result asked for) and polls (acquire) until the
// barrier's G-th arrival; the barrier's number lives in a register, so
// neither an atomic's result nor a published word lies on the way. Measured
// alone (4,000 barriers): 152 blocks of 1024 threads 1.20 us, against 1.93 us
// for an arrival that learns its barrier from the count and a last one that
// publishes its number, and 2.09 us for that with 608 blocks of 256, the same
// threads; with 608 blocks polling, the counter itself takes 2.15 us, so this
// barrier goes with few blocks per SM. The wait is bounded: the error word is
// read only while waiting, and a barrier that runs out of polls records
// kErrTimeout and ends the launch, since its block arrives nowhere again and
// the others see the error word or run out too. A grid of one block needs
// only __syncthreads.
struct GridBar {
    unsigned *count;
    int *err;
    unsigned long long limit;
    unsigned done = 0;  // barriers passed
    __device__ __forceinline__ bool sync() {
        __shared__ int s_ok;
        __syncthreads();
        if (gridDim.x == 1) return true;
        ++done;
        if (threadIdx.x == 0) {
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
            const unsigned target = done * gridDim.x;
            int ok = 1;
            unsigned long long polls = 0;
            while (bar_poll(count) < target) {
                if (++polls > limit) {
                    set_error(err, kErrTimeout);
                    ok = 0;
                    break;
                }
                if ((polls & 1023) == 0 && *((volatile int *)err) == kErrTimeout) {
                    ok = 0;
                    break;
                }
            }
            s_ok = ok;
        }
        __syncthreads();
        return s_ok != 0;
    }
};

// How a persistent sweep deals the work of one schedule step to its warps:
// the bins' units (32 vertices for the thread bin, 32 / T for a tile bin, one
// for the warp bin) follow one another round the warps, and warp numbers run
// over the blocks first, so a step of few units uses one warp on each of many
// SMs and no warp takes a second bin's unit while others have none. All warps
// of the launch count alike.
struct Deal {
    uint32_t nw, gw;     // warps of the grid, and this warp
    uint32_t next = 0;   // the warp the next bin's first unit goes to
    __device__ __forceinline__ Deal()
        : nw(gridDim.x * (blockDim.x >> 5)), gw((threadIdx.x >> 5) * gridDim.x + blockIdx.x) {}
    // this warp's first unit of the coming bin; its others follow nw apart
    __device__ __forceinline__ uint32_t first() const { return gw >= next ? gw - next : gw + nw - next; }
    __device__ __forceinline__ void pass(uint32_t units) {
        next += units;
        if (next >= nw) next %= nw;
    }
};

}  // namespace lgb
