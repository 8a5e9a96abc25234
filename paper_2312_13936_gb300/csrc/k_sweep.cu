// The sweeps' entry points: the arithmetic policy of a launch (common.cuh).
// The persistent deterministic sweep takes Det64 where the engine found
// 2m < 2^31 (c.narrow); per-step launches always take the wide policy.
#include "k_sweep_ops.h"

namespace lgb {

cudaError_t launch_sweep_eval(const SweepCtx &c, int bin, const int32_t *list, int64_t count, int max_blocks,
                              cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    return c.det ? SweepOps<Det>::eval(c, bin, list, count, max_blocks, s)
                 : SweepOps<Async>::eval(c, bin, list, count, max_blocks, s);
}
cudaError_t launch_move_apply(const SweepCtx &c, const int32_t *list, int64_t count, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    return c.det ? SweepOps<Det>::apply(c, false, list, count, s) : SweepOps<Async>::apply(c, false, list, count, s);
}
cudaError_t launch_refine_apply(const SweepCtx &c, const int32_t *list, int64_t count, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    return c.det ? SweepOps<Det>::apply(c, true, list, count, s) : SweepOps<Async>::apply(c, true, list, count, s);
}
int sweep_coop_blocks_per_sm(bool det, bool narrow, bool w_int, bool refine) {
    if (!det) return SweepOps<Async>::blocks(w_int, refine);
    return narrow ? SweepOps<Det64>::blocks(w_int, refine) : SweepOps<Det>::blocks(w_int, refine);
}
cudaError_t launch_sweep_coop(const SweepCtx &c, const int32_t *list, int grid, cudaStream_t s) {
    if (!c.det) return SweepOps<Async>::coop(c, list, grid, s);
    return c.narrow ? SweepOps<Det64>::coop(c, list, grid, s) : SweepOps<Det>::coop(c, list, grid, s);
}

}  // namespace lgb
