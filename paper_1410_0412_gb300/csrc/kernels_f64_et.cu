// Esoteric Twist steps for IEEE double grids.
#include "kernels.cuh"

namespace lbm {
LBM_INSTANTIATE_ET(LBM_F64)
}  // namespace lbm
