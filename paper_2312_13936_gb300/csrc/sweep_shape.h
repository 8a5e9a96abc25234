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

// blocks per SM of a launch: what fits, the handle's launch shape (0: no
// bound) and kCoopMaxBlocks
inline int sweep_blocks_per_sm(int fit, int32_t tuned) {
    const int b = std::min(fit, kCoopMaxBlocks);
    return tuned > 0 ? std::min<int>(b, tuned) : b;
}

// Blocks of a sweep over nsteps schedule steps of units warp units in all, of
// n vertices (vpb: leiden_tuning.vertices_per_block): enough for a step's
// work. One block (which synchronises with __syncthreads only) while its
// warps take an average step's units at once, else a block for every four
// units, and at least one for every vpb vertices. A barrier of 152 blocks
// takes 1.2 us, of 16 blocks 1.1 us, a warp's second unit 3 us and more, so
// there is little to save between one block and the full grid.
inline int sweep_grid(int per_sm, int sms, int64_t units, int32_t nsteps, int64_t n, int32_t vpb, bool grid_hubs) {
    const int64_t ups = units / nsteps;
    if (ups < 4 * (int64_t)kCoopWarps * sms) per_sm = 1;
    const int64_t full = (int64_t)per_sm * sms;
    if (grid_hubs) return (int)full;
    const int64_t want = ups <= kCoopWarps ? 1 : std::max((ups + 3) / 4, (n + vpb - 1) / vpb);
    return (int)std::max<int64_t>(1, std::min(want, full));
}

}  // namespace lgb
