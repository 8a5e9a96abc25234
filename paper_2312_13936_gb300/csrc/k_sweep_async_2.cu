#include "k_sweep.cuh"

namespace lgb {
template struct SweepOps<Async, 2>;
}  // namespace lgb
