#include "k_sweep.cuh"

namespace lgb {
template struct SweepOps<Det, 1>;
}  // namespace lgb
