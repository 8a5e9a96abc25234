#include "k_sweep.cuh"

namespace lgb {
template struct SweepOps<Async, 1>;
}  // namespace lgb
