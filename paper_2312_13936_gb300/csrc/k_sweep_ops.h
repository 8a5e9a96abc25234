// The sweeps of one arithmetic policy with MB resident blocks per SM, each
// instantiated in a translation unit of its own (k_sweep_async_1.cu, ...) from
// k_sweep.cuh so that they compile in parallel; k_sweep.cu picks one.
#pragma once
#include "common.cuh"
#include "kernels.h"

namespace lgb {

template <class P, int MB> struct SweepOps {
    // one (step, bin) of a sweep, and a step's apply phase, as launches of
    // their own (<Det, 2> and <Async, 2> only)
    static cudaError_t eval(const SweepCtx &c, int bin, const int32_t *list, int64_t count, int max_blocks,
                            cudaStream_t s);
    static cudaError_t apply(const SweepCtx &c, bool refine, const int32_t *list, int64_t count, cudaStream_t s);
    // resident blocks per SM of the persistent sweep, and its launch
    static int blocks(bool w_int, bool refine);
    static cudaError_t coop(const SweepCtx &c, const int32_t *list, int grid, cudaStream_t s);
};

}  // namespace lgb
