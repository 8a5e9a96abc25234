#include "k_sweep.cuh"

namespace lgb {
template struct SweepOps<Det, 2>;
}  // namespace lgb
