// FP64 storage and arithmetic.
#include "lbm_launchers.cuh"

namespace lbm {
LBM_INSTANTIATE(double)
}  // namespace lbm
