#include "k_sweep.cuh"

namespace lgb {
template struct SweepOps<Async>;
}  // namespace lgb
