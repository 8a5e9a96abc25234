#include "k_sweep.cuh"

namespace lgb {
template struct SweepOps<Det>;
}  // namespace lgb
