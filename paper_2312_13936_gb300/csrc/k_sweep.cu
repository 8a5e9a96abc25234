// The sweeps' entry points: the arithmetic policy of a launch (common.cuh).
// The persistent deterministic sweep takes Det64 where the engine found
// 2m < 2^31 (c.narrow), per-step launches always the wide policy; c.two: two
// blocks per SM may be resident (64 registers a thread instead of 128).
#include "k_sweep_ops.h"

namespace lgb {

cudaError_t launch_sweep_eval(const SweepCtx &c, int bin, const int32_t *list, int64_t count, int max_blocks,
                              cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    return c.det ? SweepOps<Det, 2>::eval(c, bin, list, count, max_blocks, s)
                 : SweepOps<Async, 2>::eval(c, bin, list, count, max_blocks, s);
}
cudaError_t launch_move_apply(const SweepCtx &c, const int32_t *list, int64_t count, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    return c.det ? SweepOps<Det, 2>::apply(c, false, list, count, s) : SweepOps<Async, 2>::apply(c, false, list, count, s);
}
cudaError_t launch_refine_apply(const SweepCtx &c, const int32_t *list, int64_t count, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    return c.det ? SweepOps<Det, 2>::apply(c, true, list, count, s) : SweepOps<Async, 2>::apply(c, true, list, count, s);
}
int sweep_coop_blocks_per_sm(bool det, bool narrow, bool w_int, bool refine) {
    if (!det) return SweepOps<Async, 2>::blocks(w_int, refine);
    return narrow ? SweepOps<Det64, 2>::blocks(w_int, refine) : SweepOps<Det, 2>::blocks(w_int, refine);
}
cudaError_t launch_sweep_coop(const SweepCtx &c, const int32_t *list, int grid, cudaStream_t s) {
    if (!c.det) return c.two ? SweepOps<Async, 2>::coop(c, list, grid, s) : SweepOps<Async, 1>::coop(c, list, grid, s);
    if (c.narrow)
        return c.two ? SweepOps<Det64, 2>::coop(c, list, grid, s) : SweepOps<Det64, 1>::coop(c, list, grid, s);
    return c.two ? SweepOps<Det, 2>::coop(c, list, grid, s) : SweepOps<Det, 1>::coop(c, list, grid, s);
}

}  // namespace lgb
