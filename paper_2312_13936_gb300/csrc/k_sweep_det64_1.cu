#include "k_sweep.cuh"

namespace lgb {
template struct SweepOps<Det64, 1>;
}  // namespace lgb
