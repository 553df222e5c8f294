// AA steps for double-float arithmetic on IEEE double grids.
#include "kernels.cuh"

namespace lbm {
LBM_INSTANTIATE_AA(LBM_F64_DF)
}  // namespace lbm
