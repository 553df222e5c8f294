// Esoteric Twist steps for shifted FP16 grids.
#include "kernels.cuh"

namespace lbm {
LBM_INSTANTIATE_ET(LBM_F16S)
}  // namespace lbm
