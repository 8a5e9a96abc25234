// Local-moving (Algorithm 2) and refinement (Algorithm 3) sweeps.
//
// For each vertex i the kernels accumulate K_{i->c} over the neighbour
// communities (scanCommunities / scanBounded), compute the Eq. 2 gain of
// every candidate, take the best (ties: lowest community id) and compare it
// with staying. The accumulation structure depends on the degree bin:
//   bin 1     one thread per vertex, up to 8 edges in registers, merged by
//             pairwise comparison (32 vertices per warp, 8 loads in flight each);
//   bins 2-3  a tile of 16/32 lanes holds one edge per lane; equal
//             communities find one another with one match and sum in shared
//             memory;
//   bin 4     one warp per vertex, open-addressing table in shared memory;
//   bin 5     a group of 256 threads per vertex, shared-memory table;
//   bin 6     persistent sweep: one block per vertex of up to kCtaMaxDeg
//             entries, all the block's shared memory one table; per-step
//             launches: one block per vertex, table in global memory;
//   bin 7     persistent sweep: the whole grid (longer hubs).
//
// A sweep visits the schedule steps in order (reading S0). The main kernel,
// k_sweep_coop, is persistent: one cooperative launch runs every step of a
// sweep and separates steps with a grid barrier, so a sweep costs one launch
// whatever the number of steps. Asynchronous local-moving applies each move
// at once below the capped step (atomics on Sigma, the paper's asynchronous
// execution) and records proposals in the capped steps, where neighbours
// share a step; the deterministic mode moves at once into a second copy of
// Sigma below the capped step (nothing else that a step reads is changed by
// its own moves) and records proposals from there on. An apply phase after
// the step's evaluation commits them; the refinement's
// proposals are accepted by reading S5. The per-(step, bin) kernels
// below run the same routines one launch at a time; the engine uses them if
// a cooperative launch is not possible.
//
// State that changes during a sweep (C, Sigma, sizes, flags, proposals) is
// read through L2 (ld.global.cg) so that a step sees every write made before
// the preceding barrier.
#pragma once
#include <algorithm>
#include <atomic>
#include <climits>

#include <type_traits>

#include "k_sweep_ops.h"

namespace lgb {
namespace {

template <class P, class W> struct SV {
    using A = typename P::acc;
    using T = typename P::tot;
    using S = typename P::sum;
    const int64_t *off;
    const int32_t *deg;
    const int32_t *idx;
    const W *w;
    int32_t *C;
    const int32_t *CB;
    const A *K;
    T *Sig;
    T *Sig2;       // the second copy (persistent deterministic sweep)
    int32_t *old;  // the community a vertex moved from in its step (null: no moves at once in the deterministic mode)
    int32_t *size;
    uint8_t *unproc;
    int32_t *prop;
    long long *gain;
    const int32_t *step;
    const int64_t *loff;  // rows and weights in list order (null: by vertex)
    const int32_t *lidx;
    const W *lw;
    const A *lK;
    A kscale;       // 2m (deterministic) or 1/2m (asynchronous), see move_key
    double two_m_d;
    double gamma;
    int32_t cur_step, cap_step, nsteps;
    const int64_t *key_off;
    int32_t max_it, single_sweep;
    double tau;
    T *dq_arr;                     // per-sweep gain sums (persistent phase)
    unsigned long long *moved_arr; // per-sweep refinement moves (persistent phase)
    int32_t *iters_out;
    T *dq_acc;
    unsigned long long *moved;
    int32_t *hub_keys;
    S *hub_vals;
    int hub_bits, hub_regions;
    // bin 7 on the whole grid (persistent sweep)
    const int32_t *hubs;
    const int64_t *hbase;  // ordinal of every step's first hub (null: no hubs)
    int32_t *hj;
    int64_t *htoff, *heoff, *hinfo;
    int32_t *hd, *hcand, *hmv;
    unsigned long long *hkey;
    S *hacc;                    // sums of a step's single hub by community (zero between steps)
    unsigned long long *hslot;  // every block's best candidate of a step's single hub (4 words each)
    S *hkvd;
    bool grid_hubs;
    unsigned *bar;
    int *err;
    unsigned long long *prof;
    int32_t block_max;              // rows longer than this are beyond bin 5
    int32_t stall_block;            // testing aid: this block never arrives at a barrier
    unsigned long long spin_limit;  // barrier polls before giving up
    // persistent sweep: act[k] == it + 1 marks step k as holding an eligible
    // vertex in sweep it (steps without one are skipped; the refinement from
    // its second sweep on, the local-moving of batches); null elsewhere
    int32_t *act;
    // randomized refinement (asynchronous mode): draws from SplitMix64 with
    // state rseed + 0xD1B54A32D192ED03 * (sweep + 1); sweep: the sweep of a
    // per-step launch
    bool rand_refine;
    uint64_t rseed;
    int32_t sweep;
    // batch of graphs (gid == null: one graph)
    const int32_t *gid;
    const A *gks;
    const double *g2m;
    int32_t *gdone;
    int32_t *giters;
    unsigned *gactive;
    const double *gtau;
    int32_t G;
};

// The row and weight of the vertex v at list position t: from the copy in
// list order when the pass made one (a step's rows then lie together), else
// from the vertex's own row.
template <class W> struct RowOf {
    int64_t e0;
    int32_t dv;
    const int32_t *idx;
    const W *w;
};
template <class P, class W> __device__ __forceinline__ RowOf<W> row_of(const SV<P, W> &a, int32_t v, int64_t t) {
    if (a.loff) {
        const int64_t e0 = a.loff[t];
        return {e0, (int32_t)(a.loff[t + 1] - e0), a.lidx, a.lw};
    }
    return {a.off[v], a.deg[v], a.idx, a.w};
}
template <class P, class W> __device__ __forceinline__ typename P::acc k_of(const SV<P, W> &a, int32_t v, int64_t t) {
    return a.lK ? a.lK[t] : a.K[v];
}

// A thread's sweep sums: gains or joins (asynchronous), applied gains
// (deterministic local-moving), applied proposals (refinement), and this
// sweep's per-graph slots they go to.
template <class P> struct Sums {
    GAcc<typename P::acc> gain;
    GAcc<unsigned __int128> dgain;  // deterministic gains (dq: two words per slot)
    GAcc<unsigned long long> moved;
    typename P::tot *dq;
    unsigned long long *mv;
    int32_t stamp = 0;  // this sweep's mark in act (persistent sweep)
    int32_t cur = -1;   // the step being run (persistent sweep)
    // Sigma as the step reads it and as its moves leave it: two copies in the
    // persistent deterministic sweep (see catch_up), else the same array
    typename P::tot *sr, *sw;
    // refinement: set (in shared memory) when a vertex of the step may be
    // eligible again in the next sweep (null in per-step launches)
    int *keep = nullptr;
};

template <class P, class W> SV<P, W> view(const SweepCtx &c) {
    using A = typename P::acc;
    using T = typename P::tot;
    SV<P, W> a;
    a.off = c.g.off;
    a.deg = c.g.deg;
    a.idx = c.g.idx;
    a.w = static_cast<const W *>(c.g.w);
    a.C = c.C;
    a.CB = c.CB;
    a.K = static_cast<const A *>(c.K);
    a.Sig = static_cast<T *>(c.Sig);
    a.Sig2 = P::det ? static_cast<T *>(c.Sig2) : a.Sig;
    a.old = P::det ? c.old : nullptr;
    a.size = c.size;
    a.unproc = c.unproc;
    a.prop = c.prop;
    a.gain = c.gain;
    a.step = c.step;
    a.loff = c.loff;
    a.lidx = c.lidx;
    a.lw = static_cast<const W *>(c.lw);
    a.lK = static_cast<const A *>(c.lK);
    a.kscale = P::det ? (A)c.two_m_i : (A)(1.0 / c.two_m_f);
    a.two_m_d = P::det ? (double)c.two_m_i : c.two_m_f;
    a.gamma = c.gamma;
    a.cur_step = c.cur_step;
    a.cap_step = c.cap_step;
    a.nsteps = c.nsteps;
    a.key_off = c.key_off;
    a.max_it = c.max_it;
    a.single_sweep = c.single_sweep;
    a.tau = c.tau;
    a.dq_arr = static_cast<T *>(c.dq_arr);
    a.moved_arr = c.moved_arr;
    a.iters_out = c.iters_out;
    a.dq_acc = static_cast<T *>(c.dq_acc);
    a.moved = c.moved;
    a.hub_keys = c.hub_keys;
    a.hub_vals = static_cast<typename P::sum *>(c.hub_vals);
    a.hub_bits = c.hub_bits;
    a.hub_regions = c.hub_regions;
    a.hubs = c.hubs;
    a.hbase = c.grid_hubs ? c.hbase : nullptr;
    a.hj = c.hj;
    a.htoff = c.htoff;
    a.heoff = c.heoff;
    a.hinfo = c.hinfo;
    a.hd = c.hd;
    a.hcand = c.hcand;
    a.hmv = c.hmv;
    a.hkey = c.hkey;
    a.hslot = c.hslot;
    a.hacc = static_cast<typename P::sum *>(c.hacc);
    a.hkvd = static_cast<typename P::sum *>(c.hkvd);
    a.grid_hubs = c.grid_hubs;
    a.bar = c.bar;
    a.err = c.err;
    a.prof = c.prof;
    a.block_max = c.block_max;
    a.stall_block = c.stall_block;
    a.spin_limit = c.spin_limit;
    a.act = c.act;
    a.rand_refine = c.rand_refine;
    a.rseed = c.rseed;
    a.sweep = c.sweep;
    a.gid = c.gid;
    a.gks = static_cast<const A *>(c.gks);
    a.g2m = c.g2m;
    a.gdone = c.gdone;
    a.giters = c.giters;
    a.gactive = c.gactive;
    a.gtau = c.gtau;
    a.G = c.G;
    return a;
}

__device__ __forceinline__ int32_t ldm(const int32_t *p) { return __ldcg(p); }
__device__ __forceinline__ double ldm(const double *p) { return __ldcg(p); }
__device__ __forceinline__ long long ldm(const long long *p) { return __ldcg(p); }
__device__ __forceinline__ uint8_t ldm(const uint8_t *p) { return __ldcg(p); }

// Better candidate: larger key, then smaller community id.
template <class A> __device__ __forceinline__ bool better(A k1, int32_t c1, A k2, int32_t c2) {
    return k1 > k2 || (k1 == k2 && c1 < c2);
}

// graph of vertex v and its key scale
// (B: the kernel serves a batch of graphs; the single-graph instantiations
// carry no per-graph code)
template <bool B, class P, class W> __device__ __forceinline__ int32_t graph_of(const SV<P, W> &a, int32_t v) {
    return B ? __ldg(&a.gid[v]) : 0;
}
template <bool B, class P, class W>
__device__ __forceinline__ typename P::acc kscale_of(const SV<P, W> &a, int32_t gv) {
    return B ? __ldg(&a.gks[gv]) : a.kscale;
}

// Whether a step decides by proposals that an apply phase commits after
// the step's evaluation, rather than moving at once: always in the
// deterministic mode and in the refinement, and in the asynchronous
// local-moving in the capped steps, where neighbours may share a step (on
// heavy-tailed graphs most vertices are there, and moving at once let
// neighbours chase each other).
template <class P, bool REFINE> __device__ __forceinline__ bool proposing(int32_t cur_step, int32_t cap_step) {
    return REFINE || P::det || cur_step >= cap_step;
}
// the gain of a local-moving proposal, in the key's own type (a 128-bit
// gain takes the two words gain[2v], gain[2v+1])
__device__ __forceinline__ void store_gain(long long *gain, int32_t v, __int128 g) {
    gain[2 * (int64_t)v] = (long long)(unsigned long long)g;
    gain[2 * (int64_t)v + 1] = (long long)(g >> 64);
}
__device__ __forceinline__ void store_gain(long long *gain, int32_t v, long long g) { gain[2 * (int64_t)v] = g; }
__device__ __forceinline__ void store_gain(long long *gain, int32_t v, float g) {
    reinterpret_cast<float *>(gain)[v] = g;
}
template <class K> __device__ __forceinline__ unsigned __int128 load_gain128(const long long *gain, int32_t v) {
    const unsigned long long lo = (unsigned long long)__ldcg(&gain[2 * (int64_t)v]);
    if (sizeof(K) == 8) return lo;
    const unsigned long long hi = (unsigned long long)__ldcg(&gain[2 * (int64_t)v + 1]);
    return ((unsigned __int128)hi << 64) | lo;
}

// Decision for vertex v (one thread, graph gv, key scale kscale) with best
// candidate (key, cand), K_{v->d} = kvd and Sigma_d = sd. Returns true if a
// local-moving move was made at once (its neighbours must then be marked
// unprocessed).
template <class P, class W, bool REFINE, bool B>
__device__ __forceinline__ bool decide_sd(const SV<P, W> &a, int32_t v, int32_t d, typename P::acc Kv,
                                          typename P::key key, int32_t cand, typename P::sum kvd,
                                          typename P::tot sd, Sums<P> &sm, int32_t cur_step, int32_t gv,
                                          typename P::acc kscale) {
    using A = typename P::acc;
    using T = typename P::tot;
    using K = typename P::key;
    bool mv = false;
    K g = 0;
    if (cand != INT_MAX) {
        const K ks = stay_key(kscale, kvd, Kv, sd, a.gamma);
        mv = key > ks;
        if (!REFINE && mv && cur_step >= a.cap_step) {
            // S2: where neighbours may move together, a single-vertex
            // community does not move into a larger-id single-vertex one.
            if (ldm(&a.size[d]) == 1 && ldm(&a.size[cand]) == 1 && cand > d) mv = false;
        }
        g = key - ks;
    }
    if (REFINE && sm.keep && (!mv || cur_step >= a.cap_step)) *sm.keep = 1;
    if constexpr (P::det) {
        a.prop[v] = mv ? cand : -1;
        if (a.old && cur_step < a.cap_step) {
            // Below the capped step of a persistent sweep the move is made at
            // once: no vertex of the step reads C, the size or the flags it
            // changes (they concern v's neighbours and v), and Sigma's change
            // goes to the copy the step does not read.
            if (!mv) return false;
            a.old[v] = d;
            atomic_add_acc(&sm.sw[d], -(T)Kv);
            atomic_add_acc(&sm.sw[cand], (T)Kv);
            atomicSub(&a.size[d], 1);
            atomicAdd(&a.size[cand], 1);
            a.C[v] = cand;
            if (REFINE) gacc_add(sm.moved, B, gv, 1ULL, sm.mv);
            else gacc_add(sm.dgain, B, gv, (unsigned __int128)g, reinterpret_cast<unsigned long long *>(sm.dq));
            return !REFINE;
        }
        if (!REFINE && mv) store_gain(a.gain, v, g);  // proposed: an apply phase commits
        return false;
    } else {
        if (REFINE && cur_step < a.cap_step) {
            // Asynchronous refinement below the capped step: no two vertices
            // of a step are adjacent, so the neighbour through which v saw
            // cand stays in cand and nobody joins v while it leaves: the join
            // is applied at once (the gain sum counts joins in this phase).
            if (mv) {
                atomic_add_acc(&sm.sw[d], -(T)Kv);
                atomic_add_acc(&sm.sw[cand], (T)Kv);
                atomicSub(&a.size[d], 1);
                atomicAdd(&a.size[cand], 1);
                a.C[v] = cand;
                gacc_add(sm.gain, B, gv, (A)1, sm.mv);
            }
            return false;
        }
        if (proposing<P, REFINE>(cur_step, a.cap_step)) {
            a.prop[v] = mv ? cand : -1;
            if (!REFINE && mv) store_gain(a.gain, v, g);
            return false;
        }
        if (mv) {
            atomic_add_acc(&sm.sw[d], -(T)Kv);
            atomic_add_acc(&sm.sw[cand], (T)Kv);
            atomicSub(&a.size[d], 1);
            atomicAdd(&a.size[cand], 1);
            a.C[v] = cand;
            gacc_add(sm.gain, B, gv, g, sm.dq);
        }
    }
    return mv;
}
template <class P, class W, bool REFINE, bool B>
__device__ __forceinline__ bool decide(const SV<P, W> &a, int32_t v, int32_t d, typename P::acc Kv,
                                       typename P::key key, int32_t cand, typename P::sum kvd, Sums<P> &sm,
                                       int32_t cur_step, int32_t gv, typename P::acc kscale) {
    return decide_sd<P, W, REFINE, B>(a, v, d, Kv, key, cand, kvd, ldm(&sm.sr[d]), sm, cur_step, gv, kscale);
}

// Key of candidate community c for vertex v. The randomized refinement
// (asynchronous mode) replaces the gain key > 0 of an isolated vertex (whose
// staying key is 0) by 1 / (1 - ln(U) / key), U uniform in (0, 1) from the
// vertex, the community and the sweep: the largest of these keys is a draw
// with probability proportional to the gain (Efraimidis and Spirakis'
// weighted sampling, in an order-preserving form), and it stays positive, so
// the vertex moves exactly when some gain is positive.
template <class P, class W, bool REFINE>
__device__ __forceinline__ typename P::key cand_key(const SV<P, W> &a, const Sums<P> &sm, int32_t v, int32_t c,
                                                    typename P::key kk) {
    if constexpr (P::det || !REFINE) {
        return kk;
    } else {
        if (!a.rand_refine) return kk;
        if (!(kk > 0)) return AccLimits<typename P::key>::lowest();
        const uint64_t h = splitmix64_at(a.rseed + 0xD1B54A32D192ED03ULL * (uint64_t)sm.stamp,
                                         ((uint64_t)(uint32_t)v << 32) | (uint32_t)c);
        const float u = ((float)(h >> 40) + 0.5f) * (1.0f / 16777216.0f);
        return 1.0f / (1.0f - logf(u) / kk);
    }
}

// act[k] = stamp, written only when it differs (a step's mark is read by
// many threads and written about once)
__device__ __forceinline__ void mark_step(int32_t *act, int32_t k, int32_t stamp) {
    if (__ldcg(&act[k]) != stamp) act[k] = stamp;
}
// A neighbour u of a mover becomes unprocessed (Algorithm 2 pruning); its
// step, if it is still to come in this sweep, is marked active. (A step
// before the one being run is not marked: a block that is still choosing its
// next step would take it, and meet the others at no barrier.)
template <class P, class W>
__device__ __forceinline__ void flag_unproc(const SV<P, W> &a, const Sums<P> &sm, int32_t u) {
    a.unproc[u] = 1;
    if (a.act) {
        const int32_t k = a.step[u];
        if (k > sm.cur) mark_step(a.act, k, sm.stamp);
    }
}

// Eligibility: local-moving takes unprocessed vertices and marks them
// processed (Algorithm 2 pruning); refinement takes isolated vertices (the
// community of v has v as its only member, reading R7). In a batch, the
// vertices of a graph whose phase has converged are left alone.
template <class P, class W, bool REFINE, bool B>
__device__ __forceinline__ bool take_vertex(const SV<P, W> &a, int32_t v, int32_t &d, int32_t gv) {
    if (REFINE) {
        d = ldm(&a.C[v]);
        return ldm(&a.size[d]) == 1 && !(B && ldm(&a.gdone[gv]));
    }
    d = ldm(&a.C[v]);  // in flight together with the flag
    const bool e = ldm(&a.unproc[v]) != 0 && !(B && ldm(&a.gdone[gv]));
    if (e) a.unproc[v] = 0;
    return e;
}

// --------------------------------------------------------- thread bin
// The evaluation of one eligible vertex v at list position t by its own
// thread, its row of at most E entries in registers.
template <class P, class W, bool REFINE, bool B, int E>
__device__ __forceinline__ void eval_thread(const SV<P, W> &a, int32_t v, int32_t gv, int32_t d, typename P::acc Kv,
                                            const RowOf<W> &row, int32_t cur_step, Sums<P> &sm, ProfCounts &pc) {
    using A = typename P::acc;
    using S = typename P::sum;
    const int64_t e0 = row.e0;
    const int32_t dv = row.dv;
    const typename P::tot sd = ldm(&sm.sr[d]);
    const int32_t bv = REFINE ? a.CB[v] : 0;
    int32_t jj[E];
    S wt[E];
#pragma unroll
    for (int k = 0; k < E; ++k) {
        jj[k] = -1;
        wt[k] = 0;
        if (k < dv) {
            jj[k] = row.idx[e0 + k];
            wt[k] = wconv<S>(row.w[e0 + k]);
        }
    }
    int32_t c[E];
#pragma unroll
    for (int k = 0; k < E; ++k) {
        c[k] = -1;
        bool ok = k < dv && jj[k] != v;
        if (REFINE && ok) ok = (__ldg(&a.CB[jj[k]]) == bv);
        if (ok) c[k] = ldm(&a.C[jj[k]]);
    }
    // merge equal communities into their first entry, in edge order
#pragma unroll
    for (int k = 1; k < E; ++k)
#pragma unroll
        for (int k2 = 0; k2 < k; ++k2)
            if (c[k] >= 0 && c[k2] == c[k]) {
                wt[k2] += wt[k];
                c[k] = -1;
            }
    S kvd = 0;
    typename P::key key = AccLimits<typename P::key>::lowest();
    int32_t cand = INT_MAX;
    int distinct = 0;
    const A ks = kscale_of<B>(a, gv);
#pragma unroll
    for (int k = 0; k < E; ++k) {
        if (c[k] < 0) continue;
        distinct++;
        if (c[k] == d) {
            kvd = wt[k];
            continue;
        }
        const typename P::key kk =
            cand_key<P, W, REFINE>(a, sm, v, c[k], move_key(ks, wt[k], Kv, ldm(&sm.sr[c[k]]), a.gamma));
        if (better(kk, c[k], key, cand)) {
            key = kk;
            cand = c[k];
        }
    }
    const bool mv = decide_sd<P, W, REFINE, B>(a, v, d, Kv, key, cand, kvd, sd, sm, cur_step, gv, ks);
    if (a.prof) {
        pc.v[0]++;
        pc.v[2] += dv;
        pc.v[3] += distinct;
        if (proposing<P, REFINE>(cur_step, a.cap_step) ? (a.prop[v] >= 0) : mv) {
            pc.v[4]++;
            pc.v[5] += dv;
        }
    }
    if (!REFINE && mv) {
#pragma unroll
        for (int k = 0; k < E; ++k)
            if (k < dv) flag_unproc(a, sm, jj[k]);  // neighbours (self-loop included) of a mover
    }
}

template <class P, class W, bool REFINE, bool B>
__device__ __forceinline__ void run_thread(const SV<P, W> &a, const int32_t *__restrict__ list, int64_t lo, int64_t hi,
                                           int32_t cur_step, Deal &deal, Sums<P> &sm, ProfCounts &pc) {
    const int lane = threadIdx.x & 31;
    const uint32_t units = (uint32_t)((hi - lo + 31) >> 5);
    for (uint32_t u = deal.first(); u < units; u += deal.nw) {
        const int64_t t = lo + (int64_t)u * 32 + lane;
        if (t >= hi) continue;
        const int32_t v = list[t];
        // eligibility first (Algorithm 2 pruning: the unprocessed flag;
        // refinement: the size of the vertex's community), so that a pruned
        // vertex costs one flag load and none of the header loads below
        int32_t d = 0;
        bool elig;
        if (REFINE) {
            d = ldm(&a.C[v]);
            elig = ldm(&a.size[d]) == 1;
        } else {
            elig = ldm(&a.unproc[v]) != 0;
        }
        const int32_t gv = (B && elig) ? graph_of<B>(a, v) : 0;
        if (B && elig) elig = !ldm(&a.gdone[gv]);
        if (!elig) {
            if (proposing<P, REFINE>(cur_step, a.cap_step)) a.prop[v] = -1;
            pc.v[1]++;
            continue;
        }
        if (!REFINE) {
            a.unproc[v] = 0;  // processed (Algorithm 2 pruning)
            d = ldm(&a.C[v]);
        }
        eval_thread<P, W, REFINE, B, kThreadMaxDeg>(a, v, gv, d, k_of(a, v, t), row_of(a, v, t), cur_step, sm, pc);
    }
    deal.pass(units);
}

// ----------------------------------------------------------- tile bins
// Equal communities of a tile find one another with one match instruction and
// sum in shared memory at their first lane's place (T rounds of two or three
// shuffles each, for every lane to see every other, kept the SM's one shuffle
// pipe busy: about 140 of its cycles per vertex). The vertex's header loads do
// not wait for its eligibility, and a neighbour's community not for its bound,
// far beyond L2 neither: with the eligibility first in the two-block form,
// local-moving of R-MAT of 2^25 vertices took the same 831 ms and of a
// deterministic batch of 4,096 block models 873 instead of 818; with the bound
// first, refinement 277 instead of 288 ms and 234 instead of 227.
template <class A> __device__ __forceinline__ A *tile_sums() {
    __shared__ A s_sum[kCoopWarps][32];
    return s_sum[threadIdx.x >> 5];
}
template <class P, class W, int T, bool REFINE, bool B>
__device__ __forceinline__ void run_tile(const SV<P, W> &a, const int32_t *__restrict__ list, int64_t lo, int64_t hi,
                                         int32_t cur_step, Deal &deal, Sums<P> &sm, ProfCounts &pc) {
    using A = typename P::acc;
    using S = typename P::sum;
    const int lane = threadIdx.x & 31;
    const int tl = lane & (T - 1);
    const unsigned tmask = (T == 32) ? kFull : (((1u << T) - 1u) << (lane & ~(T - 1)));
    S *wsum = tile_sums<S>();
    constexpr int per = 32 / T;  // vertices of a unit
    const uint32_t units = (uint32_t)((hi - lo + per - 1) / per);
    for (uint32_t u = deal.first(); u < units; u += deal.nw) {
        const int64_t t = lo + (int64_t)u * per + lane / T;
        if (t >= hi) continue;
        const int32_t v = list[t];
        const int32_t gv = graph_of<B>(a, v);
        const A Kv = k_of(a, v, t);
        const RowOf<W> row = row_of(a, v, t);
        const int32_t bv = REFINE ? a.CB[v] : 0;
        int32_t d = 0;
        int elig = 0;
        if (tl == 0) elig = take_vertex<P, W, REFINE, B>(a, v, d, gv) ? 1 : 0;
        elig = __shfl_sync(tmask, elig, 0, T);
        d = __shfl_sync(tmask, d, 0, T);
        if (!elig) {
            if (tl == 0 && proposing<P, REFINE>(cur_step, a.cap_step)) a.prop[v] = -1;
            if (tl == 0) pc.v[1]++;
            continue;
        }
        const int64_t e0 = row.e0;
        const int32_t dv = row.dv;
        const typename P::tot sd = ldm(&sm.sr[d]);
        int32_t j = -1, c = -1;
        S wv = 0;
        if (tl < dv) {
            j = row.idx[e0 + tl];
            wv = wconv<S>(row.w[e0 + tl]);
            c = ldm(&a.C[j]);  // beside its bound
            if (j == v || (REFINE && __ldg(&a.CB[j]) != bv)) c = -1;
        }
        // merge equal communities into their first lane's sum
        const unsigned peers = __match_any_sync(tmask, c);
        const int first = __ffs(peers) - 1;
        const bool lead = c >= 0 && first == lane;
        wsum[lane] = wv;
        __syncwarp(tmask);
        if (c >= 0 && !lead) atomic_add_acc(&wsum[first], wv);
        __syncwarp(tmask);
        const S sum = wsum[lane];
        __syncwarp(tmask);
        const unsigned dball = __ballot_sync(tmask, lead && c == d) & tmask;
        const int dsrc = dball ? ((__ffs(dball) - 1) & (T - 1)) : 0;
        const S kvd_b = __shfl_sync(tmask, sum, dsrc, T);
        const S kvd = dball ? kvd_b : (S)0;
        typename P::key key = AccLimits<typename P::key>::lowest();
        int32_t cand = INT_MAX;
        const A ks = kscale_of<B>(a, gv);
        if (lead && c != d) {
            key = cand_key<P, W, REFINE>(a, sm, v, c, move_key(ks, sum, Kv, ldm(&sm.sr[c]), a.gamma));
            cand = c;
        }
#pragma unroll
        for (int o = T / 2; o > 0; o >>= 1) {
            const typename P::key ok = kshfl_xor(tmask, key, o, T);
            const int32_t oc = __shfl_xor_sync(tmask, cand, o, T);
            if (better(ok, oc, key, cand)) {
                key = ok;
                cand = oc;
            }
        }
        int mv = 0;
        if (tl == 0) mv = decide_sd<P, W, REFINE, B>(a, v, d, Kv, key, cand, kvd, sd, sm, cur_step, gv, ks) ? 1 : 0;
        if (a.prof) {
            const unsigned lb = __ballot_sync(tmask, lead) & tmask;
            if (tl == 0) {
                pc.v[0]++;
                pc.v[2] += dv;
                pc.v[3] += __popc(lb);
                if (proposing<P, REFINE>(cur_step, a.cap_step) ? (a.prop[v] >= 0) : (mv != 0)) {
                    pc.v[4]++;
                    pc.v[5] += dv;
                }
            }
        }
        if (!REFINE) {
            mv = __shfl_sync(tmask, mv, 0, T);
            if (mv && tl < dv) flag_unproc(a, sm, j);  // neighbours (self-loop included) of a mover
        }
    }
    deal.pass(units);
}

// Entries of a row into a table by the warps of the threads ti, of stride
// threads in all: four entries of a lane in flight, each load of the chain
// (target, its bound, its community) for all four before the next. The
// weight to v's own community d stays in the lane's kvd, and communities that
// fill a good part of a warp's 32 entries are summed in the warp and added
// once: late in a phase most of a row's entries share a few communities, and
// a thousand threads' adds to one shared-memory word follow one another.
template <class P, class W, bool REFINE>
__device__ __forceinline__ void table_insert(const SV<P, W> &a, const RowOf<W> &row, int32_t v, int32_t d, int32_t bv,
                                             int ti, int stride, int32_t *keys, typename P::sum *vals, int bits,
                                             typename P::sum &kvd) {
    using S = typename P::sum;
    const int lane = threadIdx.x & 31;
    for (int32_t x0 = ti - lane; x0 < row.dv; x0 += 4 * stride) {
        int32_t j[4], c[4];
        S w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int32_t e = x0 + lane + q * stride;
            j[q] = -1;
            w[q] = 0;
            if (e < row.dv) {
                j[q] = row.idx[row.e0 + e];
                w[q] = wconv<S>(row.w[row.e0 + e]);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bool ok = j[q] >= 0 && j[q] != v;
            c[q] = ok ? ldm(&a.C[j[q]]) : -1;  // beside its bound
            if (REFINE && ok && __ldg(&a.CB[j[q]]) != bv) c[q] = -1;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (x0 + q * stride >= row.dv) break;  // the same on every lane
            if (c[q] == d) {
                kvd += w[q];
                c[q] = -1;
            }
            unsigned left = __ballot_sync(kFull, c[q] >= 0);
            for (int r = 0; r < 3 && left; ++r) {
                const int lead = __ffs(left) - 1;
                const int32_t k = __shfl_sync(kFull, c[q], lead);
                const bool mine = c[q] == k;
                const unsigned same = __ballot_sync(kFull, mine);
                if (__popc(same) < 4) break;
                const S sum = full_sum(mine ? w[q] : (S)0);
                if (lane == lead && !hash_add(keys, vals, bits, k, sum)) set_error(a.err, kErrHashFull);
                if (mine) c[q] = -1;
                left &= ~same;
            }
            if (c[q] >= 0 && !hash_add(keys, vals, bits, c[q], w[q])) set_error(a.err, kErrHashFull);
        }
    }
}
// The best candidate of a filled table over the slots first, first + stride,
// ...: four slots of a thread at a time, so that their community totals are
// in flight together.
template <class P, class W, bool REFINE>
__device__ __forceinline__ void table_best(const SV<P, W> &a, const Sums<P> &sm, int32_t v, typename P::acc Kv,
                                           typename P::acc ks, int first, int stride, int S, const int32_t *keys,
                                           const typename P::sum *vals, typename P::key &key, int32_t &cand,
                                           ProfCounts &pc) {
    for (int s0 = first; s0 < S; s0 += 4 * stride) {
        int32_t k[4];
        typename P::tot sc[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int s = s0 + q * stride;
            k[q] = s < S ? keys[s] : -1;
            sc[q] = 0;
            if (k[q] >= 0) sc[q] = ldm(&sm.sr[k[q]]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (k[q] < 0) continue;
            pc.v[3]++;
            const typename P::key kk = cand_key<P, W, REFINE>(
                a, sm, v, k[q], move_key(ks, vals[s0 + q * stride], Kv, sc[q], a.gamma));
            if (better(kk, k[q], key, cand)) {
                key = kk;
                cand = k[q];
            }
        }
    }
}

// The best candidate of a row by the threads ti of stride (keys, vals: a
// clear table of 2^bits slots; sync: their barrier). KEEP: up to four entries
// a thread, which is nearly every row, the entries stay in registers from
// their loads to their keys: a community's total is on its way while the sums
// are added, and each thread then takes the sums of its own entries' slots
// instead of scanning the table's two to four slots an entry. What a step of
// few units costs is the instructions that one warp runs one after another
// (about 11 cycles each, with 16 warps an SM of which few have work): a row
// of 37 entries spent 3,100 cycles inserting and 2,100 scanning 128 slots. The
// forms of the persistent sweep with two blocks per SM, which have 64 registers
// a thread and many units a step, go without where the four arrays spill:
// asynchronous ones stored 2.0 to 3.4 KB a thread (R-MAT of 2^25 vertices
// 2000 ms instead of 1755, a batch of 4,096 block models 1739 instead of
// 1296). Det64 spills half a KB either way and keeps its rows (the batch, in
// the deterministic mode: local-moving 818 ms, 837 without).
template <class P, class W, bool REFINE, bool KEEP, class F>
__device__ __forceinline__ void table_row(const SV<P, W> &a, const Sums<P> &sm, const RowOf<W> &row, int32_t v,
                                          int32_t d, int32_t bv, typename P::acc Kv, typename P::acc ks, int ti,
                                          int stride, int32_t *keys, typename P::sum *vals, int bits,
                                          typename P::key &key, int32_t &cand, typename P::sum &kvd, ProfCounts &pc,
                                          F &&sync) {
    using S = typename P::sum;
    if (!KEEP || row.dv > 4 * stride) {
        table_insert<P, W, REFINE>(a, row, v, d, bv, ti, stride, keys, vals, bits, kvd);
        sync();
        table_best<P, W, REFINE>(a, sm, v, Kv, ks, ti, stride, 1 << bits, keys, vals, key, cand, pc);
        return;
    }
    const int lane = threadIdx.x & 31;
    int32_t c[4], at[4];
    S w[4];
    typename P::tot sc[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int32_t e = ti + q * stride;
        c[q] = -1;
        w[q] = 0;
        at[q] = -1;
        if (e < row.dv) {
            c[q] = row.idx[row.e0 + e];
            w[q] = wconv<S>(row.w[row.e0 + e]);
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int32_t j = c[q];
        if (j < 0) continue;
        c[q] = ldm(&a.C[j]);  // beside its bound
        if (j == v || (REFINE && __ldg(&a.CB[j]) != bv)) c[q] = -1;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        sc[q] = 0;
        if (c[q] == d) {
            kvd += w[q];
            c[q] = -1;
        }
        if (c[q] >= 0) sc[q] = ldm(&sm.sr[c[q]]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (ti - lane + q * stride >= row.dv) break;  // the same on every lane
        unsigned left = __ballot_sync(kFull, c[q] >= 0);
        for (int r = 0; r < 3 && left; ++r) {  // as in table_insert
            const int lead = __ffs(left) - 1;
            const bool mine = c[q] == __shfl_sync(kFull, c[q], lead);
            const unsigned same = __ballot_sync(kFull, mine);
            if (__popc(same) < 4) break;
            const S sum = full_sum(mine ? w[q] : (S)0);
            if (lane == lead) w[q] = sum;
            else if (mine) c[q] = -1;
            left &= ~same;
        }
        if (c[q] >= 0) {
            bool fresh = false;
            at[q] = hash_slot(keys, bits, c[q], fresh);
            if (fresh) pc.v[3]++;
            if (at[q] < 0) set_error(a.err, kErrHashFull);
            else atomic_add_acc(&vals[at[q]], w[q]);
        }
    }
    sync();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (at[q] < 0) continue;
        const typename P::key kk =
            cand_key<P, W, REFINE>(a, sm, v, c[q], move_key(ks, vals[at[q]], Kv, sc[q], a.gamma));
        if (better(kk, c[q], key, cand)) {
            key = kk;
            cand = c[q];
        }
    }
}
// the best of a warp's candidates, in every lane
template <class K> __device__ __forceinline__ void warp_best(K &key, int32_t &cand) {
    for (int o = 16; o > 0; o >>= 1) {
        const K ok = kshfl_xor(kFull, key, o);
        const int32_t oc = __shfl_xor_sync(kFull, cand, o);
        if (better(ok, oc, key, cand)) {
            key = ok;
            cand = oc;
        }
    }
}

// ------------------------------------------------------- warp-table bin
template <class P, class W, bool REFINE, bool B, bool KEEP>
__device__ __forceinline__ void run_warp(const SV<P, W> &a, const int32_t *__restrict__ list, int64_t lo, int64_t hi,
                                         int32_t cur_step, int32_t *keys, typename P::sum *vals, Deal &deal,
                                         Sums<P> &sm, ProfCounts &pc) {
    using A = typename P::acc;
    const int lane = threadIdx.x & 31;
    for (int64_t t = lo + deal.first(); t < hi; t += deal.nw) {
        const int32_t v = list[t];
        const int32_t gv = graph_of<B>(a, v);
        const A Kv = k_of(a, v, t);
        const RowOf<W> row = row_of(a, v, t);
        const int32_t dv = row.dv;
        const int32_t bv = REFINE ? a.CB[v] : 0;
        int32_t d = 0;
        int elig = 0;
        if (lane == 0) elig = take_vertex<P, W, REFINE, B>(a, v, d, gv) ? 1 : 0;
        elig = __shfl_sync(kFull, elig, 0);
        d = __shfl_sync(kFull, d, 0);
        if (!elig) {
            if (lane == 0 && proposing<P, REFINE>(cur_step, a.cap_step)) a.prop[v] = -1;
            if (lane == 0) pc.v[1]++;
            continue;
        }
        int bits = ceil_log2(2 * (int64_t)dv);
        if (bits < 6) bits = 6;
        const int S = 1 << bits;
        for (int s = lane; s < S; s += 32) {
            keys[s] = -1;
            vals[s] = 0;
        }
        __syncwarp();
        const typename P::tot sd = ldm(&sm.sr[d]);
        typename P::sum kvd = 0;
        typename P::key key = AccLimits<typename P::key>::lowest();
        int32_t cand = INT_MAX;
        const A ks = kscale_of<B>(a, gv);
        table_row<P, W, REFINE, KEEP>(a, sm, row, v, d, bv, Kv, ks, lane, 32, keys, vals, bits, key, cand, kvd, pc,
                                [] { __syncwarp(); });
        warp_best(key, cand);
        kvd = full_sum(kvd);
        int mv = 0;
        if (lane == 0) {
            mv = decide_sd<P, W, REFINE, B>(a, v, d, Kv, key, cand, kvd, sd, sm, cur_step, gv, ks) ? 1 : 0;
            pc.v[0]++;
            pc.v[2] += dv;
            if (kvd != 0) pc.v[3]++;
            if (proposing<P, REFINE>(cur_step, a.cap_step) ? (a.prop[v] >= 0) : (mv != 0)) {
                pc.v[4]++;
                pc.v[5] += dv;
            }
        }
        if (!REFINE) {
            mv = __shfl_sync(kFull, mv, 0);
            if (mv)
                for (int32_t e = lane; e < dv; e += 32) flag_unproc(a, sm, row.idx[row.e0 + e]);
        }
        __syncwarp();
    }
    deal.pass((uint32_t)(hi - lo));
}

// ------------------------------------------------ block / hub table bins
// GS threads per vertex: a group of kGroup (a whole block of the per-step
// kernels, one of the groups of the persistent sweep's larger blocks, on
// named barrier 1 + the group's number) or the whole block of the persistent
// sweep. first: the group's first list position relative to lo, step: the
// number of groups. HUB: a global-memory table per block of the per-step
// kernels; only blocks below hub_regions take part.
constexpr int kMaxGroups = 4;
template <int GS> __device__ __forceinline__ void group_sync() {
    if (GS == kGroup) asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)(threadIdx.x / kGroup)), "n"(kGroup) : "memory");
    else __syncthreads();
}
template <class P, class W, bool REFINE, int GS, bool B, bool KEEP>
__device__ __forceinline__ void run_block(const SV<P, W> &a, const int32_t *__restrict__ list, int64_t lo, int64_t hi,
                                          int64_t first, int64_t step, int32_t cur_step, int32_t *keys,
                                          typename P::sum *vals, int max_bits, Sums<P> &sm, ProfCounts &pc) {
    using A = typename P::acc;
    using S = typename P::sum;
    __shared__ int ss_elig[kMaxGroups], ss_d[kMaxGroups], ss_mv[kMaxGroups];
    __shared__ typename P::key ss_key[32];
    __shared__ S ss_kvd[32];
    __shared__ int32_t ss_cand[32];
    constexpr int nw = GS >> 5;
    const int grp = threadIdx.x / GS, tid = threadIdx.x % GS, lane = tid & 31, wib = tid >> 5;
    int &s_elig = ss_elig[grp], &s_d = ss_d[grp], &s_mv = ss_mv[grp];
    typename P::key *s_key = ss_key + grp * nw;
    S *s_kvd = ss_kvd + grp * nw;
    int32_t *s_cand = ss_cand + grp * nw;
    for (int64_t t = lo + first; t < hi; t += step) {
        const int32_t v = list[t];
        const int32_t gv = graph_of<B>(a, v);
        const A Kv = k_of(a, v, t);
        const RowOf<W> row = row_of(a, v, t);
        const int32_t dv = row.dv;
        const int32_t bv = REFINE ? a.CB[v] : 0;
        int bits = ceil_log2(2 * (int64_t)dv);
        if (bits < 6) bits = 6;
        const bool fits = bits <= max_bits;
        const int Sz = fits ? 1 << bits : 0;
        // one thread takes the eligibility while the others clear the table
        if (tid == 0) {
            int32_t c = 0;
            s_elig = take_vertex<P, W, REFINE, B>(a, v, c, gv) ? 1 : 0;
            s_d = c;
        }
        for (int s = tid; s < Sz; s += GS) {
            keys[s] = -1;
            vals[s] = 0;
        }
        group_sync<GS>();
        const bool elig = s_elig != 0;
        const int32_t d = s_d;
        if (!elig || !fits) {
            if (tid == 0) {
                if (elig) set_error(a.err, kErrHashFull);
                if (proposing<P, REFINE>(cur_step, a.cap_step)) a.prop[v] = -1;
                pc.v[1]++;
            }
            group_sync<GS>();
            continue;
        }
        const typename P::tot sd = ldm(&sm.sr[d]);
        S kvd = 0;
        typename P::key key = AccLimits<typename P::key>::lowest();
        int32_t cand = INT_MAX;
        const A ks = kscale_of<B>(a, gv);
        table_row<P, W, REFINE, KEEP>(a, sm, row, v, d, bv, Kv, ks, tid, GS, keys, vals, bits, key, cand, kvd, pc,
                                [] { group_sync<GS>(); });
        warp_best(key, cand);
        kvd = full_sum(kvd);
        if (lane == 0) {
            s_key[wib] = key;
            s_cand[wib] = cand;
            s_kvd[wib] = kvd;
        }
        group_sync<GS>();
        if (wib == 0) {
            key = lane < nw ? s_key[lane] : AccLimits<typename P::key>::lowest();
            cand = lane < nw ? s_cand[lane] : INT_MAX;
            kvd = full_sum(lane < nw ? s_kvd[lane] : (S)0);
            warp_best(key, cand);
            if (lane == 0) {
                s_mv =
                    decide_sd<P, W, REFINE, B>(a, v, d, Kv, key, cand, kvd, sd, sm, cur_step, gv, ks) ? 1 : 0;
                pc.v[0]++;
                prof_add(a.prof, 2, dv);
                if (kvd != 0) pc.v[3]++;
                if (proposing<P, REFINE>(cur_step, a.cap_step) ? (a.prop[v] >= 0) : (s_mv != 0)) {
                    pc.v[4]++;
                    prof_add(a.prof, 5, dv);
                }
            }
        }
        if (!REFINE) {
            group_sync<GS>();
            if (s_mv)
                for (int64_t e = tid; e < dv; e += GS) flag_unproc(a, sm, row.idx[row.e0 + e]);
        }
    }
    group_sync<GS>();
}

// -------------------------------------------- bin 7 on the whole grid
// In the persistent sweep the vertices of bin 7 (rows of more than
// kCtaMaxDeg entries) of a step are evaluated by every block together:
// degree-first schedules put a few hubs in each of many steps, and one block
// per hub would leave the rest of the GPU waiting on the largest. Hub j of
// the pass (its ordinal in list order) is hubs[j]. Phases, each ended by a
// grid barrier: block 0 takes the eligibility of the step's hubs and lays
// out the eligible ones (hj[p] = j; table slots [htoff[p], htoff[p+1]), a
// power of two of at least 2 deg; row entries [heoff[p], heoff[p+1]) of the
// flat walk); clearing; insertion of the rows (entries of one warp step
// with equal (hub, community) summed first); the largest key per hub
// (atomicMax on an order-preserving encoding); the smallest community id
// among those with that key (atomicMin), which is the candidate a block's
// own scan finds; the decision, one thread per hub; for an asynchronous
// local-moving move, the neighbours' flags. A step whose hubs are all
// ineligible ends after the first phase.
// order-preserving unsigned encodings of the keys: a 128-bit key as (high
// word with its sign bit flipped, low word), compared high word first; a
// 64-bit key as one word; an fp32 key in the low 32 bits
__device__ __forceinline__ void key_order(__int128 k, unsigned long long &hi, unsigned long long &lo) {
    hi = (unsigned long long)(long long)(k >> 64) ^ 0x8000000000000000ULL;
    lo = (unsigned long long)k;
}
__device__ __forceinline__ __int128 key_of_order(unsigned long long hi, unsigned long long lo, __int128) {
    return (__int128)(((unsigned __int128)(hi ^ 0x8000000000000000ULL) << 64) | lo);
}
__device__ __forceinline__ void key_order(long long k, unsigned long long &hi, unsigned long long &lo) {
    hi = (unsigned long long)k ^ 0x8000000000000000ULL;
    lo = 0ULL;
}
__device__ __forceinline__ long long key_of_order(unsigned long long hi, unsigned long long, long long) {
    return (long long)(hi ^ 0x8000000000000000ULL);
}
__device__ __forceinline__ void key_order(float k, unsigned long long &hi, unsigned long long &lo) {
    const unsigned u = __float_as_uint(k);
    hi = (unsigned long long)((u & 0x80000000u) ? ~u : (u | 0x80000000u));
    lo = 0ULL;
}
__device__ __forceinline__ float key_of_order(unsigned long long e, unsigned long long, float) {
    const unsigned u = (unsigned)e;
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// the p in [0, np) whose range [off[p], off[p+1]) holds x (off ascending)
__device__ __forceinline__ int64_t range_at(const int64_t *off, int64_t np, int64_t x) {
    int64_t lo = 0, hi = np - 1;  // the last p with off[p] <= x
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (__ldcg(&off[mid]) <= x) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// exclusive block scan of x (every thread of the block calls it); returns
// the block total in *total
__device__ __forceinline__ long long block_scan_excl(long long x, long long *total) {
    __shared__ long long s_w[32];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, nw = blockDim.x >> 5;
    long long inc = x;
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += y;
    }
    __syncthreads();
    if (lane == 31) s_w[wib] = inc;
    __syncthreads();
    long long before = 0, all = 0;
    for (int w = 0; w < nw; ++w) {
        if (w < wib) before += s_w[w];
        all += s_w[w];
    }
    *total = all;
    return before + inc - x;
}

// The neighbours of the step's moving hubs become unprocessed (Algorithm 2
// pruning), the whole grid walking the hubs' rows as one flat range (the
// layout of run_hubs_grid: eligible hub p owns entries [heoff[p],
// heoff[p+1]) of hub hj[p]). A hub moved when hmv[j] is set (a move made at
// once) or, in an apply phase (by_prop), when its proposal is set.
template <class P, class W>
__device__ __forceinline__ void hub_flags(const SV<P, W> &a, const Sums<P> &sm, int64_t np, int64_t E, bool by_prop) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    // a contiguous range of entries per warp, following the hub as it goes
    // (a row is longer than 32 entries: 32 consecutive ones span at most two)
    const int64_t per = ((E + warps - 1) / warps + 31) & ~(int64_t)31;
    const int64_t x1 = (gw + 1) * per < E ? (gw + 1) * per : E;
    if (gw * per >= x1) return;
    int64_t p = 0;
    if (lane == 0) p = range_at(a.heoff, np, gw * per);
    p = __shfl_sync(kFull, p, 0);
    int64_t nb = __ldcg(&a.heoff[p + 1]);
    for (int64_t x0 = gw * per; x0 < x1; x0 += 32) {
        while (x0 >= nb) nb = __ldcg(&a.heoff[++p + 1]);
        const int64_t x = x0 + lane;
        if (x >= x1) continue;
        const int64_t pl = x >= nb ? p + 1 : p;
        const int64_t j = __ldcg(&a.hj[pl]);
        const int32_t v = __ldg(&a.hubs[j]);
        if (by_prop ? (ldm(&a.prop[v]) < 0) : !__ldcg(&a.hmv[j])) continue;
        flag_unproc(a, sm, a.idx[a.off[v] + (x - __ldcg(&a.heoff[pl]))]);
    }
}

// the packed whole-grid hub tables (asynchronous mode, Det64): one 8-byte word
// per slot (key and fp32 or 32-bit integer sum, hash_add_kv) in the value
// buffer, which holds 8 bytes per slot
template <class P, class W> __device__ __forceinline__ unsigned long long *hub_kv(const SV<P, W> &a) {
    return reinterpret_cast<unsigned long long *>(a.hub_vals);
}

template <class P, class W, bool REFINE, bool B>
__device__ __forceinline__ bool run_hubs_grid(const SV<P, W> &a, int64_t j0, int64_t nh, int32_t cur_step,
                                              GridBar &bar, Sums<P> &sm, ProfCounts &pc) {
    using S = typename P::sum;
    const int lane = threadIdx.x & 31;
    const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t warps = nthreads >> 5, gw = tid >> 5;
    int64_t np, slots, E;
    {
        // eligibility and layout (block 0)
        if (blockIdx.x == 0) {
            long long np = 0, ns = 0, ne = 0;
            for (int64_t i0 = 0; i0 < nh; i0 += blockDim.x) {
                const int64_t i = i0 + threadIdx.x;
                bool e = false;
                int64_t sz = 0, dv = 0;
                if (i < nh) {
                    const int64_t j = j0 + i;
                    const int32_t v = __ldg(&a.hubs[j]);
                    const int32_t gv = graph_of<B>(a, v);
                    int32_t d = 0;
                    e = take_vertex<P, W, REFINE, B>(a, v, d, gv);
                    if (!e) {
                        if (proposing<P, REFINE>(cur_step, a.cap_step)) a.prop[v] = -1;
                        pc.v[1]++;
                    } else {
                        dv = a.deg[v];
                        int bits = ceil_log2(2 * dv);
                        if (bits < 6) bits = 6;
                        sz = 1LL << bits;
                        if (P::det) {
                            a.hkey[2 * j] = 0ULL;
                            a.hkey[2 * j + 1] = 0ULL;
                        } else {
                            a.hkey[j] = 0ULL;
                        }
                        a.hcand[j] = INT_MAX;
                        a.hkvd[j] = 0;
                        a.hmv[j] = 0;
                    }
                    a.hd[j] = e ? d : -1;
                }
                long long tp, ts, te;
                const long long p = block_scan_excl(e ? 1 : 0, &tp);
                const long long so = block_scan_excl(sz, &ts);
                const long long eo = block_scan_excl(dv, &te);
                if (e) {
                    a.hj[np + p] = (int32_t)(j0 + i);
                    a.htoff[np + p] = ns + so;
                    a.heoff[np + p] = ne + eo;
                }
                np += tp;
                ns += ts;
                ne += te;
            }
            if (threadIdx.x == 0) {
                a.htoff[np] = ns;
                a.heoff[np] = ne;
                a.hinfo[0] = np;
                a.hinfo[1] = ns;
                a.hinfo[2] = ne;
            }
        }
        if (!bar.sync()) return false;
        np = __ldcg(&a.hinfo[0]);
        slots = __ldcg(&a.hinfo[1]);
        E = __ldcg(&a.hinfo[2]);
        if (np == 0) return true;
    }
    // Each warp takes one contiguous range of entries (insertion) or slots
    // (key passes), 32 at a time, and follows the hub they belong to as it
    // goes: one binary search at the start of its range, then a step to the
    // next hub when a boundary is passed. A hub's row is longer than 32
    // entries, so 32 consecutive entries span at most two hubs; its table is
    // a power of two of at least 8192 slots, so 32 aligned slots lie in one.
    // insertion (the tables are clean: the last scan of a step clears every
    // slot it reads, and the engine clears them before the first sweep)
    {
        const int64_t per = ((E + warps - 1) / warps + 31) & ~(int64_t)31;
        const int64_t x1 = (gw + 1) * per < E ? (gw + 1) * per : E;
        int64_t p = 0, nb = 0;  // hub of the warp's current entry and the end of its row
        if (gw * per < x1) {
            if (lane == 0) p = range_at(a.heoff, np, gw * per);
            p = __shfl_sync(kFull, p, 0);
            nb = __ldcg(&a.heoff[p + 1]);
        }
        for (int64_t x0 = gw * per; x0 < x1; x0 += 32) {
            while (x0 >= nb) nb = __ldcg(&a.heoff[++p + 1]);  // the same on every lane
            const int64_t x = x0 + lane;
            const int64_t pl = x >= nb ? p + 1 : p;
            int32_t key = -1, bits = 0;
            int64_t tbase = 0;
            S val = 0;
            if (x < x1) {
                const int32_t v = __ldg(&a.hubs[__ldcg(&a.hj[pl])]);
                const int64_t e = a.off[v] + (x - (pl == p ? nb - a.deg[v] : nb));
                const int32_t u = a.idx[e];
                if (u != v && (!REFINE || __ldg(&a.CB[u]) == __ldg(&a.CB[v]))) {
                    key = ldm(&a.C[u]);
                    val = wconv<S>(a.w[e]);
                    tbase = __ldcg(&a.htoff[pl]);
                    bits = __ffsll((long long)(__ldcg(&a.htoff[pl + 1]) - tbase)) - 1;
                }
            }
            const unsigned long long pair = key >= 0 ? ((unsigned long long)pl << 32) | (uint32_t)key : ~0ULL;
            const unsigned peers = __match_any_sync(kFull, pair);
            val = peer_sum(peers, val);
            if (key >= 0 && lane == __ffs(peers) - 1) {
                bool ok;
                if constexpr (!P::packed) ok = hash_add(a.hub_keys + tbase, a.hub_vals + tbase, bits, key, val);
                else ok = hash_add_kv(hub_kv<P>(a) + tbase, bits, key, val);
                if (!ok) set_error(a.err, kErrHashFull);
            }
        }
    }
    if (!bar.sync()) return false;
    // deterministic mode: the largest key per hub -- a 128-bit key's high
    // word (pass 0), then its low word among the slots with that high word
    // (pass 1) -- then the smallest community id with that key; asynchronous
    // mode: one pass, key and id packed in one word (fp32 key above the
    // complemented id, so that the largest word is the largest key with the
    // smallest id). K_{v->d} from the slot of v's own community. The last
    // pass clears the slots. The lanes of a warp read one hub's table, so
    // each pass needs one reduction over the warp and one atomic.
    constexpr int npass = !P::det ? 1 : P::packed ? 2 : 3;
    constexpr int Q = 4;  // slots per lane and iteration: 128 aligned slots lie in one table
    using T = typename P::tot;
    const int64_t sper = ((slots + warps - 1) / warps + 32 * Q - 1) & ~(int64_t)(32 * Q - 1);
    const int64_t s1 = (gw + 1) * sper < slots ? (gw + 1) * sper : slots;
    for (int pass = 0; pass < npass; ++pass) {
        int64_t p = 0, nb = 0;  // table of the warp's current slots and its end
        if (gw * sper < s1) {
            if (lane == 0) p = range_at(a.htoff, np, gw * sper);
            p = __shfl_sync(kFull, p, 0);
            nb = __ldcg(&a.htoff[p + 1]);
        }
        int64_t j = -1;
        int32_t d = -1, v = 0;
        typename P::acc kv = 0, ks = 0;
        unsigned long long hhi = 0, hlo = 0;  // the hub's largest key so far (passes 1 and 2)
        for (int64_t s0 = gw * sper; s0 < s1; s0 += 32 * Q) {
            if (s0 >= nb || j < 0) {  // the warp enters a table: its hub's constants
                while (s0 >= nb) nb = __ldcg(&a.htoff[++p + 1]);
                j = __ldcg(&a.hj[p]);
                d = __ldcg(&a.hd[j]);
                v = __ldg(&a.hubs[j]);
                kv = a.K[v];
                ks = kscale_of<B>(a, graph_of<B>(a, v));
                if (P::det && pass > 0) {
                    hhi = __ldcg(&a.hkey[2 * j]);
                    hlo = __ldcg(&a.hkey[2 * j + 1]);
                }
            }
            // the lane's slots s0 + lane + 32 q: keys first, then the sums
            // and the candidates' totals, all loads of a round in flight
            int32_t kq[Q];
            S vq[Q];
            T sq[Q];
            if constexpr (!P::packed) {
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const int64_t sl = s0 + 32 * q + lane;
                    kq[q] = sl < s1 ? __ldcg(&a.hub_keys[sl]) : -1;
                }
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    vq[q] = 0;
                    if (kq[q] >= 0) vq[q] = __ldcg(&a.hub_vals[s0 + 32 * q + lane]);
                }
            } else {  // key and value in one word
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const int64_t sl = s0 + 32 * q + lane;
                    const unsigned long long kv = sl < s1 ? __ldcg(&hub_kv<P>(a)[sl]) : kEmptyKV;
                    kq[q] = (int32_t)(uint32_t)kv;
                    kv_value(kv, vq[q]);
                }
            }
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                sq[q] = 0;
                if (kq[q] >= 0 && kq[q] != d) sq[q] = ldm(&sm.sr[kq[q]]);
            }
            unsigned long long lmax = 0ULL;
            int32_t lmin = INT_MAX;
            bool any = false;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int32_t k = kq[q];
                if (k < 0) continue;
                if (pass == npass - 1) {
                    if constexpr (!P::packed) {
                        a.hub_keys[s0 + 32 * q + lane] = -1;
                        a.hub_vals[s0 + 32 * q + lane] = 0;
                    } else {
                        hub_kv<P>(a)[s0 + 32 * q + lane] = kEmptyKV;
                    }
                }
                if (k == d) {
                    if (pass == 0) a.hkvd[j] = vq[q];
                    continue;
                }
                unsigned long long enc, enc_lo;
                key_order(cand_key<P, W, REFINE>(a, sm, v, k, move_key(ks, vq[q], kv, sq[q], a.gamma)), enc, enc_lo);
                if (!P::det) enc = (enc << 32) | (unsigned long long)(~(uint32_t)k);
                any = true;
                if (pass == 0) {
                    pc.v[3]++;
                    lmax = enc > lmax ? enc : lmax;
                } else if (npass == 3 && pass == 1) {
                    if (enc == hhi) lmax = enc_lo > lmax ? enc_lo : lmax;
                } else if (enc == hhi && (npass < 3 || enc_lo == hlo)) {
                    lmin = k < lmin ? k : lmin;
                }
            }
            if (!__any_sync(kFull, any)) continue;
            if (pass == 0 || (npass == 3 && pass == 1)) {
                // the largest high word (pass 0), the largest low word among
                // the slots with the hub's largest high word (pass 1)
                for (int o = 16; o > 0; o >>= 1) {
                    const unsigned long long y = __shfl_xor_sync(kFull, lmax, o);
                    lmax = y > lmax ? y : lmax;
                }
                if (lane == 0) {
                    if (pass == 0) atomicMax(&a.hkey[P::det ? 2 * j : j], lmax);
                    else if (lmax) atomicMax(&a.hkey[2 * j + 1], lmax);
                }
            } else {
                for (int o = 16; o > 0; o >>= 1) {
                    const int32_t y = __shfl_xor_sync(kFull, lmin, o);
                    lmin = y < lmin ? y : lmin;
                }
                if (lane == 0 && lmin != INT_MAX) atomicMin(&a.hcand[j], lmin);
            }
        }
        if (!bar.sync()) return false;
    }
    // decisions
    for (int64_t p = tid; p < np; p += nthreads) {
        const int64_t j = __ldcg(&a.hj[p]);
        const int32_t d = __ldcg(&a.hd[j]);
        const int32_t v = __ldg(&a.hubs[j]);
        const int32_t gv = graph_of<B>(a, v);
        using K = typename P::key;
        int32_t c;
        K bk;
        if (P::det) {
            c = __ldcg(&a.hcand[j]);
            bk = c == INT_MAX ? AccLimits<K>::lowest()
                              : key_of_order(__ldcg(&a.hkey[2 * j]), __ldcg(&a.hkey[2 * j + 1]), K(0));
        } else {
            const unsigned long long best = __ldcg(&a.hkey[j]);
            c = best == 0ULL ? INT_MAX : (int32_t)~(uint32_t)best;
            bk = best == 0ULL ? AccLimits<K>::lowest() : key_of_order(best >> 32, 0ULL, K(0));
        }
        const S kd = __ldcg(&a.hkvd[j]);
        const bool mv = decide<P, W, REFINE, B>(a, v, d, a.K[v], bk, c, kd, sm, cur_step, gv, kscale_of<B>(a, gv));
        const int32_t dv = a.deg[v];
        pc.v[0]++;
        prof_add(a.prof, 2, dv);
        if (proposing<P, REFINE>(cur_step, a.cap_step) ? (ldm(&a.prop[v]) >= 0) : mv) {
            pc.v[4]++;
            prof_add(a.prof, 5, dv);
        }
        if (!REFINE && mv) a.hmv[j] = 1;
    }
    if (!REFINE && cur_step < a.cap_step) {
        // a local-moving move made at once flags the hub's neighbours
        if (!bar.sync()) return false;
        hub_flags<P, W>(a, sm, np, E, false);
    }
    return true;
}

// A layered step (below cap_step: no two of its vertices are adjacent) with
// one such hub, as most steps of a heavy-tailed schedule have: two grid
// barriers here and the step's own end. One thread of every block reads the
// hub's eligibility -- no vertex of the step can change it (a flag is set, or
// a community joined, only by a neighbour), and the barriers of the previous
// step made its last writes visible. Chunks of 32 entries go round the warps
// after the step's smaller units. The sums K_{v->c} are added, without asking
// for a result, into a vector addressed by community (hacc, zero between
// steps); after the first barrier the same chunks read the sum and the
// community's total of their entries, so the row is its own list of
// candidates: no table is probed (a chain of up to a dozen L2 atomics at half
// load) and no empty slots are scanned, and C of a hub's neighbours does not
// change within the step. Each block reduces its best candidate and leaves it
// in its own word; after the second barrier every block reduces those words
// and knows the decision (the hub's own sum and total are read between the
// barriers, where nothing writes them), so the neighbours' flags need no
// barrier of their own, and the chunks clear the sums. Block 0 makes the
// move.
// False when a barrier ran out.
template <class P, class W, bool REFINE, bool B>
__device__ __forceinline__ bool run_hub_single(const SV<P, W> &a, int64_t j0, int32_t cur_step, GridBar &bar,
                                              Deal &deal, Sums<P> &sm, ProfCounts &pc) {
    using A = typename P::acc;
    using S = typename P::sum;
    using T = typename P::tot;
    using K = typename P::key;
    __shared__ unsigned long long s_hi[32], s_lo[32];
    __shared__ int32_t s_c[32];
    __shared__ int s_moves, s_e;
    __shared__ int32_t s_d;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const bool first_thread = blockIdx.x == 0 && threadIdx.x == 0;
    const int32_t v = __ldg(&a.hubs[j0]);
    const int32_t gv = graph_of<B>(a, v);
    if (threadIdx.x == 0) {
        s_d = ldm(&a.C[v]);
        bool x = REFINE ? ldm(&a.size[s_d]) == 1 : ldm(&a.unproc[v]) != 0;
        if (B && x) x = !ldm(&a.gdone[gv]);
        s_e = x ? 1 : 0;
    }
    const int64_t e0 = a.off[v];
    const int32_t dv = a.deg[v];
    const int32_t bv = REFINE ? __ldg(&a.CB[v]) : 0;
    // the entry of chunk i in this lane: its vertex (-1: none) and community
    // (-1: not a candidate)
    auto entry = [&](uint32_t i, int32_t &u, int32_t &c) {
        const int64_t x = (int64_t)i * 32 + lane;
        u = x < dv ? a.idx[e0 + x] : -1;
        c = u >= 0 ? ldm(&a.C[u]) : -1;
        if (u == v || (REFINE && u >= 0 && __ldg(&a.CB[u]) != bv)) c = -1;
    };
    const uint32_t chunks = ((uint32_t)dv + 31) / 32, i0 = deal.first();
    int32_t u0 = -1, c0 = -1;  // the warp's first chunk stays in registers; it loads beside the eligibility
    S w0 = 0;
    if (i0 < chunks) {
        entry(i0, u0, c0);
        if (u0 >= 0) w0 = wconv<S>(a.w[e0 + (int64_t)i0 * 32 + lane]);
    }
    __syncthreads();
    const int32_t d = s_d;
    if (!s_e) {  // the same in every block
        if (first_thread) {
            if (proposing<P, REFINE>(cur_step, a.cap_step)) a.prop[v] = -1;
            pc.v[1]++;
        }
        return true;
    }
    for (uint32_t i = i0; i < chunks; i += deal.nw) {
        int32_t u = u0, c = c0;
        S val = w0;
        if (i != i0) {
            entry(i, u, c);
            val = u >= 0 ? wconv<S>(a.w[e0 + (int64_t)i * 32 + lane]) : (S)0;
        }
        if (c < 0) val = 0;
        const unsigned peers = __match_any_sync(kFull, c);
        val = peer_sum(peers, val);
        if (c >= 0 && lane == __ffs(peers) - 1) {
            atomic_add_acc(&a.hacc[c], val);
            pc.v[3]++;
        }
    }
    deal.pass(chunks);
    if (!bar.sync()) return false;
    if (!REFINE && first_thread) a.unproc[v] = 0;  // every block has read the flag
    const T sd = ldm(&sm.sr[d]);
    const S kd = __ldcg(&a.hacc[d]);
    const A kv = a.K[v], ks = kscale_of<B>(a, gv);
    K key = AccLimits<K>::lowest();
    int32_t cand = INT_MAX;
    for (uint32_t i = i0; i < chunks; i += deal.nw) {
        int32_t u = u0, c = c0;
        if (i != i0) entry(i, u, c);
        if (c < 0 || c == d) continue;
        const S sum = __ldcg(&a.hacc[c]);
        const K kk = cand_key<P, W, REFINE>(a, sm, v, c, move_key(ks, sum, kv, ldm(&sm.sr[c]), a.gamma));
        if (better(kk, c, key, cand)) {
            key = kk;
            cand = c;
        }
    }
    warp_best(key, cand);
    if (lane == 0) {
        key_order(key, s_hi[wib], s_lo[wib]);
        s_c[wib] = cand;
    }
    __syncthreads();
    if (wib == 0) {
        const bool in = lane < (int)(blockDim.x >> 5);
        key = in ? key_of_order(s_hi[lane], s_lo[lane], K(0)) : AccLimits<K>::lowest();
        cand = in ? s_c[lane] : INT_MAX;
        warp_best(key, cand);
        if (lane == 0) {
            unsigned long long *slot = a.hslot + 4 * (size_t)blockIdx.x;
            unsigned long long hi, lo;
            key_order(key, hi, lo);
            slot[0] = hi;
            slot[1] = lo;
            slot[2] = (unsigned long long)(uint32_t)cand;
        }
    }
    if (!bar.sync()) return false;
    if (wib == 0) {
        key = AccLimits<K>::lowest();
        cand = INT_MAX;
        for (unsigned b = lane; b < gridDim.x; b += 32) {
            const unsigned long long *slot = a.hslot + 4 * (size_t)b;
            const unsigned long long hi = __ldcg(&slot[0]), lo = __ldcg(&slot[1]);
            const int32_t c = (int32_t)(uint32_t)__ldcg(&slot[2]);
            const K k = key_of_order(hi, lo, K(0));
            if (c != INT_MAX && better(k, c, key, cand)) {
                key = k;
                cand = c;
            }
        }
        warp_best(key, cand);
        if (lane == 0) {
            const bool mv = cand != INT_MAX && key > stay_key(ks, kd, kv, sd, a.gamma);
            s_moves = mv ? 1 : 0;
            if (blockIdx.x == 0) {
                decide_sd<P, W, REFINE, B>(a, v, d, kv, key, cand, kd, sd, sm, cur_step, gv, ks);
                pc.v[0]++;
                prof_add(a.prof, 2, dv);
                if (mv) {
                    pc.v[4]++;
                    prof_add(a.prof, 5, dv);
                }
            }
        }
    }
    if (!REFINE) __syncthreads();
    const bool flag = !REFINE && s_moves;
    for (uint32_t i = i0; i < chunks; i += deal.nw) {
        int32_t u = u0, c = c0;
        if (i != i0) entry(i, u, c);
        if (c >= 0) a.hacc[c] = 0;
        if (flag && u >= 0) flag_unproc(a, sm, u);
    }
    return true;
}

// ------------------------------------------------------------ apply steps
// vertices of a warp's unit in an apply phase: 32 when the step has work for
// every warp, fewer (the other lanes then only help with the rows) when more
// warps would stand idle
__device__ __forceinline__ int apply_unit(uint32_t count, uint32_t nw) {
    return count > 16 * nw ? 32 : count > 4 * nw ? 8 : 2;
}

// The persistent deterministic sweep keeps two copies of Sigma, so that a
// layered step needs one grid barrier: the step reads one copy (sr) while its
// moves change the other (sw), and the copies change places at its end. What
// a step's moves wrote is missing from the copy it read; the next step, which
// does not read that copy, adds it there (the vertices of [lo, hi) that moved
// in their step: prop, from old). The sums are integers, so the order in
// which the two steps' changes arrive does not matter. (With proposals that
// an apply phase committed, every layered step took two barriers and walked
// its movers' rows a second time for their flags.)
template <class P, class W>
__device__ __forceinline__ void catch_up(const SV<P, W> &a, const int32_t *__restrict__ list, int64_t lo, int64_t hi,
                                         Deal &deal, const Sums<P> &sm) {
    const int lane = threadIdx.x & 31;
    const int per = apply_unit((uint32_t)(hi - lo), deal.nw);
    const uint32_t units = (uint32_t)((hi - lo + per - 1) / per);
    for (uint32_t u = deal.first(); u < units; u += deal.nw) {
        const int64_t t = lo + (int64_t)u * per + lane;
        if (lane >= per || t >= hi) continue;
        const int32_t v = list[t];
        const int32_t c = ldm(&a.prop[v]), d = ldm(&a.old[v]);
        if (c < 0) continue;
        const auto Kv = (typename P::tot)k_of(a, v, t);
        atomic_add_acc(&sm.sw[d], -Kv);
        atomic_add_acc(&sm.sw[c], Kv);
    }
    deal.pass(units);
}

// Commits the proposal of list position t (v = -1: none) and returns v's row
// (empty when v stays).
template <class P, class W, bool B>
__device__ __forceinline__ RowOf<W> commit_move(const SV<P, W> &a, int32_t v, int64_t t, Sums<P> &sm) {
    const int32_t c = v >= 0 ? ldm(&a.prop[v]) : -1;
    if (c < 0) return {0, 0, nullptr, nullptr};
    const int32_t d = ldm(&a.C[v]);
    const auto Kv = (typename P::tot)k_of(a, v, t);
    atomic_add_acc(&sm.sr[d], -Kv);
    atomic_add_acc(&sm.sr[c], Kv);
    if (P::det && sm.sw != sm.sr) {
        atomic_add_acc(&sm.sw[d], -Kv);
        atomic_add_acc(&sm.sw[c], Kv);
    }
    atomicSub(&a.size[d], 1);
    atomicAdd(&a.size[c], 1);
    a.C[v] = c;
    if (P::det)
        gacc_add(sm.dgain, B, graph_of<B>(a, v), load_gain128<typename P::key>(a.gain, v),
                 reinterpret_cast<unsigned long long *>(sm.dq));
    else
        gacc_add(sm.gain, B, graph_of<B>(a, v),
                 (typename P::acc)__ldcg(reinterpret_cast<const float *>(a.gain) + v), sm.dq);
    return row_of(a, v, t);
}

// Proposals of one capped step (of any step in the per-step launches of the
// deterministic mode): commit them and flag the movers' neighbours.
// [lo, mid): rows of up to kFlat entries (longer ones among them go to a warp
// each): the movers' rows of a unit are flagged as one flat range of entries
// by all lanes, four loads per lane in flight (a lane walking its own mover's
// row waited for every load in turn: 16 us a step on a 200,000-vertex block
// model with rows of 24 entries). [mid, flags): a vertex a warp (32 rows of
// thousands of entries in one warp's unit kept the grid waiting for 260 us a
// step on R-MAT 1M). [flags, hi): the commit alone (their neighbours are
// flagged by hub_flags over the step's hub layout).
template <class P, class W, bool B>
__device__ __forceinline__ void run_move_apply(const SV<P, W> &a, const int32_t *__restrict__ list, int64_t lo,
                                               int64_t mid, int64_t flags, int64_t hi, Deal &deal, Sums<P> &sm) {
    constexpr int32_t kFlat = 1024;
    const int lane = threadIdx.x & 31;
    const int32_t *is = a.loff ? a.lidx : a.idx;
    // row entries [e0, e0 + dv) by the whole warp
    auto flag_row = [&](int64_t e0, int32_t dv) {
        for (int32_t x = 0; x < dv; x += 128) {
            int32_t j[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) j[q] = x + 32 * q + lane < dv ? is[e0 + x + 32 * q + lane] : -1;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (j[q] >= 0) flag_unproc(a, sm, j[q]);
        }
    };
    const int per = apply_unit((uint32_t)(mid - lo), deal.nw);
    const uint32_t units = (uint32_t)((mid - lo + per - 1) / per);
    for (uint32_t u = deal.first(); u < units; u += deal.nw) {
        const int64_t t = lo + (int64_t)u * per + lane;
        const RowOf<W> row = commit_move<P, W, B>(a, lane < per && t < mid ? list[t] : -1, t, sm);
        if (!__any_sync(kFull, row.dv > 0)) continue;
        const int32_t flat = row.dv <= kFlat ? row.dv : 0;
        int32_t incl = flat;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        const int32_t total = __shfl_sync(kFull, incl, 31);
        const int64_t base = row.e0 - (incl - flat);  // entry x of the flat range is is[base + x] of its owner
        for (int32_t x0 = 0; x0 < total; x0 += 128) {
            int32_t j[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int32_t x = x0 + 32 * q + lane;
                int own = 0;  // lanes whose rows end at or before x
#pragma unroll
                for (int st = 16; st >= 1; st >>= 1)
                    if (__shfl_sync(kFull, incl, own + st - 1) <= x) own += st;
                const int64_t bs = __shfl_sync(kFull, base, own & 31);
                j[q] = x < total ? is[bs + x] : -1;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (j[q] >= 0) flag_unproc(a, sm, j[q]);
        }
        unsigned longs = __ballot_sync(kFull, row.dv > kFlat);
        while (longs) {
            const int src = __ffs(longs) - 1;
            longs &= longs - 1;
            flag_row(__shfl_sync(kFull, row.e0, src), __shfl_sync(kFull, row.dv, src));
        }
    }
    deal.pass(units);
    for (int64_t t = mid + deal.first(); t < hi; t += deal.nw) {
        RowOf<W> row{0, 0, nullptr, nullptr};
        if (lane == 0) row = commit_move<P, W, B>(a, list[t], t, sm);
        if (t < flags) flag_row(__shfl_sync(kFull, row.e0, 0), __shfl_sync(kFull, row.dv, 0));
    }
    deal.pass((uint32_t)(hi - mid));
}

// Refinement: accept proposal v -> t unless t is a single-vertex community
// whose vertex proposes in the same step; of a mutual pair the larger id
// moves (reading S5). Accepted vertices join t.
template <class P, class W, bool B>
__device__ __forceinline__ void run_refine_apply(const SV<P, W> &a, const int32_t *__restrict__ list, int64_t lo,
                                                 int64_t hi, int32_t cur_step, Deal &deal, Sums<P> &sm) {
    const int lane = threadIdx.x & 31;
    const int per = apply_unit((uint32_t)(hi - lo), deal.nw);
    const uint32_t units = (uint32_t)((hi - lo + per - 1) / per);
    for (uint32_t u = deal.first(); u < units; u += deal.nw) {
        const int64_t t = lo + (int64_t)u * per + lane;
        if (lane >= per || t >= hi) continue;
        const int32_t v = list[t];
        const int32_t tg = ldm(&a.prop[v]);
        if (tg < 0) continue;
        const int32_t pt = (__ldg(&a.step[tg]) == cur_step) ? ldm(&a.prop[tg]) : -1;
        if (!(pt < 0 || (pt == v && v > tg))) continue;
        const auto Kv = (typename P::tot)k_of(a, v, t);
        atomic_add_acc(&sm.sr[v], -Kv);
        atomic_add_acc(&sm.sr[tg], Kv);
        if (P::det && sm.sw != sm.sr) {
            atomic_add_acc(&sm.sw[v], -Kv);
            atomic_add_acc(&sm.sw[tg], Kv);
        }
        atomicSub(&a.size[v], 1);
        atomicAdd(&a.size[tg], 1);
        a.C[v] = tg;
        gacc_add(sm.moved, B, graph_of<B>(a, v), 1ULL, sm.mv);
    }
    deal.pass(units);
}

// ------------------------------------------------------- persistent sweep
// Blocks of 512 threads, one per SM while an average step has fewer than four
// units for each of their warps, else two (sweep_shape.h): a step of few units
// costs with the arrivals at its barrier and with the instructions of warps
// that have nothing to do, a step of many with the loads in flight. (R-MAT 1M,
// one block of 1024 threads 242.0 ms, of 512 229.9 ms when this was chosen. One
// block of 512 threads or two, of the present kernels: asynchronous R-MAT of
// 2^23 vertices 632 and 536 ms, of 2^22 370 and 345; deterministic 831 and 749,
// 449 and 451.) Both forms are compiled (MB blocks per SM), so that the one
// block has 128 registers a thread and the table bins nothing to spill.
constexpr int kCoopThreads = 32 * kCoopWarps;
static_assert(kCoopThreads / kGroup <= kMaxGroups && kCoopThreads % kGroup == 0, "groups of the block bin");
static_assert(kCtaSlots <= kBlockSlots * (kCoopThreads / kGroup), "the block's table lies in its groups' tables");

// a sweep's gain sum of graph g: two words per slot (deterministic, 128 bits)
// or one fp64 word
__device__ __forceinline__ double gain_sum(long long *dq, int64_t g) {
    const unsigned long long *w = reinterpret_cast<const unsigned long long *>(dq) + 2 * g;
    return u128_words_to_double(__ldcg(&w[0]), __ldcg(&w[1]));
}
__device__ __forceinline__ double gain_sum(double *dq, int64_t g) { return __ldcg(&dq[g]); }

// shared-memory tables of every group of kGroup threads: 8 warp tables of
// kWarpSlots slots, or one block table of kBlockSlots slots (values first,
// then keys)
template <class A> __host__ __device__ constexpr size_t table_bytes() { return (sizeof(A) + sizeof(int32_t)) * kBlockSlots; }
template <class A> __device__ __forceinline__ A *table_vals() {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    return reinterpret_cast<A *>(smem_raw + (threadIdx.x / kGroup) * table_bytes<A>());
}
template <class A> __device__ __forceinline__ int32_t *table_keys() {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    return reinterpret_cast<int32_t *>(smem_raw + (threadIdx.x / kGroup) * table_bytes<A>() +
                                       sizeof(A) * kBlockSlots);
}
// the same space as one table of kCtaSlots slots for the whole block
template <class A> __device__ __forceinline__ A *cta_vals() {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    return reinterpret_cast<A *>(smem_raw);
}
template <class A> __device__ __forceinline__ int32_t *cta_keys() {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    return reinterpret_cast<int32_t *>(smem_raw + sizeof(A) * kCtaSlots);
}

// One whole phase: sweeps until the phase converges -- local-moving stops
// when a sweep's delta-modularity (reading S4 for the deterministic mode) is
// at most tau (Algorithm 2), refinement when a sweep moves nobody (reading
// R6) -- or max_it sweeps ran. The test reads per-sweep sums after a grid
// barrier, so every block takes the same decision. In a batch every graph
// takes the test on its own sums; the phase ends when no graph is left.
template <class P, class W, bool REFINE, bool B, int MB>
__global__ void __launch_bounds__(kCoopThreads, MB) k_sweep_coop(SV<P, W> a, const int32_t *__restrict__ list) {
    static_assert(MB <= kCoopMaxBlocks, "scratch of the blocks of a launch");
    using A = typename P::acc;
    using T = typename P::tot;
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    using S = typename P::sum;
    int32_t *skeys = table_keys<S>();
    S *svals = table_vals<S>();
    const int wslot = (wib & (kGroup / 32 - 1)) * kWarpSlots;  // the warp's table in its group's
    constexpr bool batch = B;
    constexpr bool KEEP = MB == 1 || std::is_same_v<P, Det64>;  // table_row
    // testing aid: this block ends without arriving at any barrier, so the
    // others' bounded wait runs out (kErrTimeout) and the launch ends
    if ((int32_t)blockIdx.x == a.stall_block) return;
    __shared__ int64_t s_ko[2][kNumBins + 2];
    __shared__ int32_t s_next;
    __shared__ int s_keep;
    if (threadIdx.x == 0) s_keep = 0;
    GridBar bar{a.bar, a.err, a.spin_limit};
    Deal deal;
    ProfCounts pc;
    int32_t it = 0;
    bool ok = true;
    while (ok && it < a.max_it) {
        Sums<P> sm;
        sm.dq = a.dq_arr + (size_t)it * a.G * (P::det ? 2 : 1);  // deterministic: two words per slot
        sm.mv = a.moved_arr + (size_t)it * a.G;
        sm.stamp = it + 1;
        sm.sr = a.Sig;
        sm.sw = a.Sig2;
        int64_t late0 = 0, late1 = 0;  // the step whose moves sw lacks (catch_up)
        if (REFINE && a.act) sm.keep = &s_keep;
        // Steps without an eligible vertex are passed over where a.act says
        // so (act[k] == the sweep's stamp: step k holds one). In the
        // refinement a vertex stays eligible only by staying isolated, so a
        // step's own evaluation in one sweep marks it for the next (all steps
        // run in the first); without the marks the sweeps after the first, in
        // which few vertices or none are left, took every step's barrier.
        const bool pick = a.act && (!REFINE || it > 0);
        // (two sets of marks by sweep in the refinement: a block may mark a
        // step for the next sweep while another still looks for it in this one)
        const int32_t *act_now = REFINE ? a.act + (it & 1) * kActSteps : a.act;
        int32_t *act_next = REFINE ? a.act + ((it + 1) & 1) * kActSteps : nullptr;
        if (!REFINE && a.act) {
            // local-moving of a batch: steps holding an unprocessed vertex at
            // the start of the sweep; moves mark the steps of the neighbours
            // they flag as the sweep goes on
            const int64_t nl = __ldcg(&a.key_off[(int64_t)a.nsteps * kNumBins]);
            for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nl;
                 t += (int64_t)gridDim.x * blockDim.x) {
                const int32_t v = list[t];
                if (B && ldm(&a.gdone[graph_of<B>(a, v)])) continue;
                if (ldm(&a.unproc[v]) != 0) mark_step(a.act, a.step[v], sm.stamp);
            }
            if (!(ok = bar.sync())) break;
        }
        // A step's nine (step, bin) offsets and the ordinal of its first hub
        // go to shared memory by lanes of warp 0, for the next step while
        // this one runs: two buffers, the other one free since the barrier
        // that ended the step before.
        auto load_ko = [&](int32_t k) -> int64_t {
            if (lane <= kNumBins) return __ldg(&a.key_off[(int64_t)k * kNumBins + lane]);
            return (lane == kNumBins + 1 && a.hbase) ? __ldg(&a.hbase[k]) : 0;
        };
        if (wib == 0 && !pick && lane <= kNumBins + 1) s_ko[0][lane] = load_ko(0);
        __syncthreads();
        int buf = 0;
        for (int32_t k = 0; k < a.nsteps && ok; ++k, buf ^= 1) {
            int64_t *sko = s_ko[buf];
            int64_t ahead = 0;
            if (pick) {
                // the next step marked as holding an eligible vertex: the
                // same in every block, since marks are only set before the
                // barrier that ended the last step taken
                if (wib == 0) {
                    int32_t n = k;
                    for (; n < a.nsteps; n += 32) {
                        const unsigned m =
                            __ballot_sync(kFull, n + lane < a.nsteps && __ldcg(&act_now[n + lane]) == sm.stamp);
                        if (m) {
                            n += __ffs(m) - 1;
                            break;
                        }
                    }
                    if (n < a.nsteps && lane <= kNumBins + 1) sko[lane] = load_ko(n);
                    if (lane == 0) s_next = n;
                }
                __syncthreads();
                k = s_next;
                if (k >= a.nsteps) break;
            } else if (wib == 0 && k + 1 < a.nsteps) {
                ahead = load_ko(k + 1);
            }
            auto fetched = [&]() {
                if (wib == 0 && !pick && k + 1 < a.nsteps && lane <= kNumBins + 1) s_ko[buf ^ 1][lane] = ahead;
            };
            const int64_t b0 = sko[0], b8 = sko[8];
            if (b0 == b8) {  // empty step: every block sees the same counts
                fetched();
                __syncthreads();
                continue;
            }
            sm.cur = k;
            const int64_t b2 = sko[2], b3 = sko[3], b4 = sko[4], b5 = sko[5], b6 = sko[6], b7 = sko[7];
            if (b2 > b0) run_thread<P, W, REFINE, B>(a, list, b0, b2, k, deal, sm, pc);
            if (b3 > b2) run_tile<P, W, 16, REFINE, B>(a, list, b2, b3, k, deal, sm, pc);
            if (b4 > b3) run_tile<P, W, 32, REFINE, B>(a, list, b3, b4, k, deal, sm, pc);
            if (b5 > b4) run_warp<P, W, REFINE, B, KEEP>(a, list, b4, b5, k, skeys + wslot, svals + wslot, deal, sm, pc);
            if (b7 > b5) {
                // rows of up to kBlockMaxDeg entries: a group each, or a
                // whole block each while the step has no more of them than
                // there are blocks; longer ones, up to kCtaMaxDeg, a block
                const bool blocks = b6 - b5 <= (int64_t)gridDim.x;
                const int64_t turn = (blockIdx.x + gridDim.x - deal.next % gridDim.x) % gridDim.x;
                if (b6 > b5 && !blocks) {
                    group_sync<kGroup>();  // the group's warp tables become one block table
                    run_block<P, W, REFINE, kGroup, B, KEEP>(a, list, b5, b6,
                                                       (int64_t)(threadIdx.x / kGroup) * gridDim.x + blockIdx.x,
                                                       (int64_t)gridDim.x * (kCoopThreads / kGroup), k, skeys, svals,
                                                       ceil_log2(kBlockSlots), sm, pc);
                }
                if (blocks || b7 > b6) {
                    __syncthreads();  // all tables become one
                    run_block<P, W, REFINE, kCoopThreads, B, KEEP>(a, list, blocks ? b5 : b6, b7, turn, gridDim.x, k,
                                                             cta_keys<S>(), cta_vals<S>(), ceil_log2(kCtaSlots), sm,
                                                             pc);
                }
                deal.pass((uint32_t)((b7 - b5) % gridDim.x));
            }
            if (P::det && late1 > late0) catch_up<P, W>(a, list, late0, late1, deal, sm);
            bool hub_layout = false;  // run_hubs_grid laid out this step's hubs
            if (b8 > b7) {
                if (b8 - b7 == 1 && k < a.cap_step) {
                    ok = run_hub_single<P, W, REFINE, B>(a, sko[kNumBins + 1], k, bar, deal, sm, pc);
                } else {
                    ok = run_hubs_grid<P, W, REFINE, B>(a, sko[kNumBins + 1], b8 - b7, k, bar, sm, pc);
                    hub_layout = true;
                }
                if (!ok) break;
            }
            fetched();
            if (REFINE && a.act) {
                // one store a block marks the step for the next sweep
                __syncthreads();
                if (threadIdx.x == 0 && s_keep) {
                    act_next[k] = sm.stamp + 1;
                    s_keep = 0;
                }
            }
            if (!(ok = bar.sync())) break;
            // a layered step's moves are made; an apply phase commits the
            // proposals where neighbours may share a step
            late0 = late1 = 0;
            if (k >= a.cap_step) {
                if (REFINE) {
                    run_refine_apply<P, W, B>(a, list, b0, b8, k, deal, sm);
                } else {
                    run_move_apply<P, W, B>(a, list, b0, b5, hub_layout ? b7 : b8, b8, deal, sm);
                    if (hub_layout) hub_flags<P, W>(a, sm, __ldcg(&a.hinfo[0]), __ldcg(&a.hinfo[2]), true);
                }
                if (!(ok = bar.sync())) break;
            } else if (P::det) {
                late0 = b0;
                late1 = b8;
                typename P::tot *const sr = sm.sr;
                sm.sr = sm.sw;
                sm.sw = sr;
            }
        }
        if (!ok) break;
        if (P::det && late1 > late0) catch_up<P, W>(a, list, late0, late1, deal, sm);  // both copies are whole
        // this sweep's sums: one graph reduces per warp, a batch flushes
        // every thread's running sum into its graph's slot
        if (batch) {
            if (REFINE) {
                if (!P::det) gacc_flush(sm.gain, sm.mv);
                gacc_flush(sm.moved, sm.mv);
            } else if (P::det) {
                gacc_flush(sm.dgain, reinterpret_cast<unsigned long long *>(sm.dq));
            } else {
                gacc_flush(sm.gain, sm.dq);
            }
        } else if (REFINE) {
            unsigned long long moved = sm.moved.v;
            if (!P::det) moved += (unsigned long long)(sm.gain.v + (A)0.5);
            moved = warp_sum(moved);
            if (lane == 0 && moved) atomicAdd(&sm.mv[0], moved);
        } else if (P::det) {
            const unsigned __int128 g = warp_sum_u128(sm.dgain.v);
            if (lane == 0 && g) atomic_add_u128(reinterpret_cast<unsigned long long *>(sm.dq), g);
        } else {
            const A g = warp_sum(sm.gain.v);
            if (lane == 0 && g != (A)0) atomic_add_acc(&sm.dq[0], (T)g);
        }
        if (!(ok = bar.sync())) break;
        bool stop;
        if (batch) {
            // every graph still running takes its own test; graphs that
            // stop record their sweep count, the others are counted
            unsigned running = 0;
            for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < a.G;
                 g += (int64_t)gridDim.x * blockDim.x) {
                if (__ldcg(&a.gdone[g])) continue;
                bool sg;
                if (REFINE) {
                    sg = __ldcg(&sm.mv[g]) == 0ULL || a.single_sweep;
                } else {
                    const double tm = a.g2m[g];
                    const double sum = gain_sum(sm.dq, g);
                    // a graph without edges (2m = 0) has nothing to move
                    const double tau = a.gtau ? a.gtau[g] : a.tau;
                    sg = !(tm > 0) || (P::det ? 2.0 * sum / (tm * tm) : 2.0 * sum / tm) <= tau;
                }
                if (sg) {
                    a.gdone[g] = 1;
                    a.giters[g] = it + 1;
                } else {
                    running++;
                }
            }
            running = warp_sum(running);
            if (lane == 0 && running) atomicAdd(&a.gactive[it], running);
            if (!(ok = bar.sync())) break;
            stop = __ldcg(&a.gactive[it]) == 0u;
        } else if (REFINE) {
            stop = __ldcg(&sm.mv[0]) == 0ULL || a.single_sweep;
        } else {
            // sweep delta-modularity from the summed gains: 2 num / (2m)^2
            // (deterministic, reading S4) or 2 sum / 2m (asynchronous)
            const double tm = a.two_m_d;
            const double sum = gain_sum(sm.dq, 0);
            const double dq = P::det ? 2.0 * sum / (tm * tm) : 2.0 * sum / tm;
            stop = dq <= a.tau;
        }
        ++it;
        if (stop) break;
    }
    if (batch) {
        // graphs still running when the phase ends ran every sweep
        for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < a.G; g += (int64_t)gridDim.x * blockDim.x)
            if (!__ldcg(&a.gdone[g])) a.giters[g] = it;
    } else if (blockIdx.x == 0 && threadIdx.x == 0 && a.giters) {
        a.giters[0] = it;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.iters_out = it;
    pc.flush(a.prof);
}

// ------------------------------------------- one (step, bin) per launch
// (one graph only) local-moving gains into the sweep's delta-modularity sum;
// asynchronous refinement joins into the move count
template <class P, class W> __device__ __forceinline__ Sums<P> scalar_sums(const SV<P, W> &a) {
    Sums<P> sm;
    sm.dq = a.dq_acc;
    sm.mv = a.moved;
    sm.stamp = a.sweep + 1;
    sm.sr = sm.sw = a.Sig;
    return sm;
}
template <class P, class W, bool REFINE>
__device__ __forceinline__ void flush_gain(const SV<P, W> &a, Sums<P> &sm) {
    using A = typename P::acc;
    if (P::det) return;
    if (REFINE) {
        const unsigned long long c = warp_sum((unsigned long long)(sm.gain.v + (A)0.5));
        if ((threadIdx.x & 31) == 0 && c) atomicAdd(a.moved, c);
    } else {
        const A s = warp_sum(sm.gain.v);
        if ((threadIdx.x & 31) == 0 && s != (A)0) atomic_add_acc(a.dq_acc, (typename P::tot)s);
    }
}

template <class P, class W, bool REFINE>
__global__ void __launch_bounds__(256) k_eval_thread(SV<P, W> a, const int32_t *__restrict__ list, int64_t count) {
    Sums<P> sm = scalar_sums(a);
    ProfCounts pc;
    Deal deal;
    run_thread<P, W, REFINE, false>(a, list, 0, count, a.cur_step, deal, sm, pc);
    flush_gain<P, W, REFINE>(a, sm);
    pc.flush(a.prof);
}
template <class P, class W, int T, bool REFINE>
__global__ void __launch_bounds__(256) k_eval_tile(SV<P, W> a, const int32_t *__restrict__ list, int64_t count) {
    Sums<P> sm = scalar_sums(a);
    ProfCounts pc;
    Deal deal;
    run_tile<P, W, T, REFINE, false>(a, list, 0, count, a.cur_step, deal, sm, pc);
    flush_gain<P, W, REFINE>(a, sm);
    pc.flush(a.prof);
}
template <class P, class W, bool REFINE>
__global__ void __launch_bounds__(256) k_eval_warp(SV<P, W> a, const int32_t *__restrict__ list, int64_t count) {
    using A = typename P::acc;
    using S = typename P::sum;
    int32_t *skeys = table_keys<S>();
    S *svals = table_vals<S>();
    const int wib = threadIdx.x >> 5;
    Sums<P> sm = scalar_sums(a);
    ProfCounts pc;
    Deal deal;
    run_warp<P, W, REFINE, false, true>(a, list, 0, count, a.cur_step, skeys + wib * kWarpSlots, svals + wib * kWarpSlots,
                                  deal, sm, pc);
    flush_gain<P, W, REFINE>(a, sm);
    pc.flush(a.prof);
}
template <class P, class W, bool REFINE, bool HUB>
__global__ void __launch_bounds__(256) k_eval_block(SV<P, W> a, const int32_t *__restrict__ list, int64_t count) {
    using A = typename P::acc;
    using S = typename P::sum;
    int32_t *skeys = table_keys<S>();
    S *svals = table_vals<S>();
    Sums<P> sm = scalar_sums(a);
    ProfCounts pc;
    if (HUB) {
        const int64_t base = (int64_t)blockIdx.x << a.hub_bits;
        if ((int64_t)blockIdx.x < (int64_t)a.hub_regions)
            run_block<P, W, REFINE, kGroup, false, true>(a, list, 0, count, blockIdx.x, a.hub_regions, a.cur_step,
                                                   a.hub_keys + base, a.hub_vals + base, a.hub_bits, sm, pc);
    } else {
        run_block<P, W, REFINE, kGroup, false, true>(a, list, 0, count, blockIdx.x, gridDim.x, a.cur_step, skeys, svals,
                                               ceil_log2(kBlockSlots), sm, pc);
    }
    flush_gain<P, W, REFINE>(a, sm);
    pc.flush(a.prof);
}
template <class P, class W>
__global__ void __launch_bounds__(256) k_move_apply(SV<P, W> a, const int32_t *__restrict__ list, int64_t count) {
    Sums<P> sm = scalar_sums(a);
    Deal deal;
    run_move_apply<P, W, false>(a, list, 0, count, count, count, deal, sm);
    if (P::det) {
        const unsigned __int128 g = warp_sum_u128(sm.dgain.v);
        if ((threadIdx.x & 31) == 0 && g) atomic_add_u128(reinterpret_cast<unsigned long long *>(a.dq_acc), g);
    } else {
        flush_gain<P, W, false>(a, sm);
    }
}
template <class P, class W>
__global__ void __launch_bounds__(256) k_refine_apply(SV<P, W> a, const int32_t *__restrict__ list, int64_t count) {
    Sums<P> sm = scalar_sums(a);
    Deal deal;
    run_refine_apply<P, W, false>(a, list, 0, count, a.cur_step, deal, sm);
    const unsigned long long mv = warp_sum(sm.moved.v);
    if ((threadIdx.x & 31) == 0 && mv) atomicAdd(a.moved, mv);
}

// raise the dynamic shared-memory limit of a kernel (a host-side attribute:
// cheap, and set before every launch so no kernel can miss it)
template <class K> cudaError_t allow_table_smem(K kern, size_t bytes) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <class P, class W, bool REFINE>
cudaError_t eval_typed(const SweepCtx &c, int bin, const int32_t *list, int64_t count, int max_blocks,
                       cudaStream_t s) {
    SV<P, W> a = view<P, W>(c);
    constexpr size_t tb = table_bytes<typename P::sum>();
    auto grid = [&](int64_t per_block) {
        int64_t b = (count + per_block - 1) / per_block;
        return (int)(b < max_blocks ? (b < 1 ? 1 : b) : max_blocks);
    };
    switch (bin) {
        case 1: k_eval_thread<P, W, REFINE><<<grid(256), 256, 0, s>>>(a, list, count); break;
        case 2: k_eval_tile<P, W, 16, REFINE><<<grid(16), 256, 0, s>>>(a, list, count); break;
        case 3: k_eval_tile<P, W, 32, REFINE><<<grid(8), 256, 0, s>>>(a, list, count); break;
        case 4: {
            cudaError_t e = allow_table_smem(k_eval_warp<P, W, REFINE>, tb);
            if (e != cudaSuccess) return e;
            k_eval_warp<P, W, REFINE><<<grid(8), 256, tb, s>>>(a, list, count);
            break;
        }
        case 5: {
            cudaError_t e = allow_table_smem(k_eval_block<P, W, REFINE, false>, tb);
            if (e != cudaSuccess) return e;
            k_eval_block<P, W, REFINE, false><<<grid(1), 256, tb, s>>>(a, list, count);
            break;
        }
        case 6:
            a.hub_regions = max_blocks;
            k_eval_block<P, W, REFINE, true><<<grid(1), 256, 0, s>>>(a, list, count);
            break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <class P, class W>
cudaError_t eval_mode(const SweepCtx &c, int bin, const int32_t *list, int64_t count, int max_blocks, cudaStream_t s) {
    return c.refine ? eval_typed<P, W, true>(c, bin, list, count, max_blocks, s)
                    : eval_typed<P, W, false>(c, bin, list, count, max_blocks, s);
}

int apply_grid(int64_t count) {
    int64_t b = (count + 255) / 256;
    return (int)(b < 1 ? 1 : (b > 4096 ? 4096 : b));
}

template <class P, class W, bool REFINE, bool B, int MB>
cudaError_t coop_launch(const SweepCtx &c, const int32_t *list, int grid, cudaStream_t s) {
    SV<P, W> a = view<P, W>(c);
    constexpr size_t all = table_bytes<typename P::sum>() * (kCoopThreads / kGroup);
    cudaError_t e = allow_table_smem(k_sweep_coop<P, W, REFINE, B, MB>, all);
    if (e != cudaSuccess) return e;
    // without a row beyond the tile bins no table is used: the L1 keeps the space
    const size_t tb = c.tables ? all : 0;
    void *args[] = {&a, (void *)&list};
    return cudaLaunchCooperativeKernel((const void *)k_sweep_coop<P, W, REFINE, B, MB>, dim3(grid), dim3(kCoopThreads),
                                       args, tb, s);
}
template <class P, class W, bool REFINE, int MB>
cudaError_t coop_typed(const SweepCtx &c, const int32_t *list, int grid, cudaStream_t s) {
    return c.gid ? coop_launch<P, W, REFINE, true, MB>(c, list, grid, s) : coop_launch<P, W, REFINE, false, MB>(c, list, grid, s);
}
template <class P, class W, bool REFINE, bool B, int MB> int coop_blocks_b() {
    constexpr size_t tb = table_bytes<typename P::sum>() * (kCoopThreads / kGroup);
    if (allow_table_smem(k_sweep_coop<P, W, REFINE, B, MB>, tb) != cudaSuccess) return 0;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sweep_coop<P, W, REFINE, B, MB>, kCoopThreads, tb) !=
        cudaSuccess)
        return 0;
    return per_sm;
}
template <class P, class W, bool REFINE, int MB> int coop_blocks_typed() {
    // both forms share the launch bounds; take the smaller occupancy (kept once
    // known: several calls of every pass need it; a query that failed is asked
    // again, so that one failure does not leave a process without the kernel)
    static std::atomic<int> known{0};
    int blocks = known.load(std::memory_order_relaxed);
    if (blocks <= 0) {
        blocks = std::min(coop_blocks_b<P, W, REFINE, false, MB>(), coop_blocks_b<P, W, REFINE, true, MB>());
        if (blocks > 0) known.store(blocks, std::memory_order_relaxed);
    }
    return blocks;
}

}  // namespace

template <class P, int MB>
cudaError_t SweepOps<P, MB>::eval(const SweepCtx &c, int bin, const int32_t *list, int64_t count, int max_blocks,
                              cudaStream_t s) {
    if constexpr (MB == 1 || std::is_same_v<P, Det64>) return cudaErrorInvalidValue;  // per-step launches take <Det, 2>, <Async, 2>
    else if constexpr (P::det)
        return c.g.w_int ? eval_mode<P, WInt>(c, bin, list, count, max_blocks, s)
                         : eval_mode<P, float>(c, bin, list, count, max_blocks, s);
    else return eval_mode<P, float>(c, bin, list, count, max_blocks, s);
}
template <class P, int MB>
cudaError_t SweepOps<P, MB>::apply(const SweepCtx &c, bool refine, const int32_t *list, int64_t count, cudaStream_t s) {
    if constexpr (MB == 1 || std::is_same_v<P, Det64>) return cudaErrorInvalidValue;
    else {
        const int g = apply_grid(count);
        if (P::det && c.g.w_int) {
            if constexpr (P::det) {
                if (refine) k_refine_apply<P, WInt><<<g, 256, 0, s>>>(view<P, WInt>(c), list, count);
                else k_move_apply<P, WInt><<<g, 256, 0, s>>>(view<P, WInt>(c), list, count);
            }
        } else {
            if (refine) k_refine_apply<P, float><<<g, 256, 0, s>>>(view<P, float>(c), list, count);
            else k_move_apply<P, float><<<g, 256, 0, s>>>(view<P, float>(c), list, count);
        }
        return cudaGetLastError();
    }
}
template <class P, int MB> int SweepOps<P, MB>::blocks(bool w_int, bool refine) {
    if constexpr (P::det)
        if (w_int) return refine ? coop_blocks_typed<P, WInt, true, MB>() : coop_blocks_typed<P, WInt, false, MB>();
    return refine ? coop_blocks_typed<P, float, true, MB>() : coop_blocks_typed<P, float, false, MB>();
}
template <class P, int MB>
cudaError_t SweepOps<P, MB>::coop(const SweepCtx &c, const int32_t *list, int grid, cudaStream_t s) {
    if constexpr (P::det)
        if (c.g.w_int)
            return c.refine ? coop_typed<P, WInt, true, MB>(c, list, grid, s) : coop_typed<P, WInt, false, MB>(c, list, grid, s);
    return c.refine ? coop_typed<P, float, true, MB>(c, list, grid, s) : coop_typed<P, float, false, MB>(c, list, grid, s);
}

}  // namespace lgb
