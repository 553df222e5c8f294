// AA steps for IEEE double grids.
#include "kernels.cuh"

namespace lbm {
LBM_INSTANTIATE_AA(LBM_F64)
}  // namespace lbm
