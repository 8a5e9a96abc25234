// The launch shape of a persistent sweep (host only; no CUDA).
#pragma once
#include <algorithm>
#include <cstdint>

namespace lgb {

constexpr int kCoopWarps = 16;     // warps of a persistent sweep's block
// Resident blocks per SM of a persistent sweep, at most: the two compiled
// forms are bounded for one and two, and a launch's scratch (a word group of
// a single hub's candidate for every block) is sized for two, whatever more
// the occupancy of a form would allow.
constexpr int kCoopMaxBlocks = 2;

// A sweep's work, step by step: its steps that have any, their warp units, and
// the rounds one block's warps would take over them.
struct SweepWork {
    int64_t units = 0, rounds = 0, steps = 0;
    void step(int64_t u) {
        if (u <= 0) return;
        units += u;
        rounds += (u + kCoopWarps - 1) / kCoopWarps;
        ++steps;
    }
};

// Blocks of a sweep of n vertices, at most fit per SM (tuned, vpb:
// leiden_tuning.coop_blocks_per_sm, vertices_per_block): enough for a step's
// work. A barrier of 152 blocks takes 1.2 us, of 16 blocks 1.1 us, a warp's
// second unit 3 us and more, so there is little to save between one block and
// the full grid. One block, which synchronises with __syncthreads only, while
// the rounds it takes beyond the first of every step cost less than the
// barriers it saves (the steps one by one: the average over the layers of a
// clique of 1,000 and the wide steps of 230,000 lattice vertices around it puts
// the wide ones on one SM, 113.9 ms a deterministic run instead of 94.5); else
// a block for every four units of an average step, and at least one for every
// vpb vertices, up to one or two per SM, as the handle's launch shape says: by
// default one while an average step holds fewer than four units for each of
// their warps (128 registers a thread instead of 64 shorten the chain of a step
// of few units; more loads in flight win where there are many).
inline int sweep_grid(int fit, int32_t tuned, int sms, const SweepWork &w, int64_t n, int32_t vpb, bool grid_hubs) {
    const int64_t ups = w.steps > 0 ? w.units / w.steps : 0;
    const int most = tuned > 0 ? tuned : ups < 4 * (int64_t)kCoopWarps * sms ? 1 : kCoopMaxBlocks;
    const int per_sm = std::min({fit, most, kCoopMaxBlocks});
    const int64_t full = (int64_t)per_sm * sms;
    if (grid_hubs) return (int)full;
    const int64_t want =
        3 * (w.rounds - w.steps) <= w.steps ? 1 : std::max((ups + 3) / 4, (n + vpb - 1) / vpb);
    return (int)std::max<int64_t>(1, std::min(want, full));
}

}  // namespace lgb
