// AA steps for single grids.
#include "kernels.cuh"

namespace lbm {
LBM_INSTANTIATE_AA(LBM_F32)
}  // namespace lbm
