// State set-up and read-back kernels, one instantiation per storage precision
// (double-float grids are IEEE double).
#include "kernels.cuh"

namespace lbm {
LBM_INSTANTIATE_STATE(LBM_F64)
LBM_INSTANTIATE_STATE(LBM_F32)
LBM_INSTANTIATE_STATE(LBM_F16S)
}  // namespace lbm
