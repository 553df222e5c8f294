// Esoteric Twist steps for single grids.
#include "kernels.cuh"

namespace lbm {
LBM_INSTANTIATE_ET(LBM_F32)
}  // namespace lbm
