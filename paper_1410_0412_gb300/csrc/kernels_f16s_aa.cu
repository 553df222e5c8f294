// AA steps for shifted FP16 grids.
#include "kernels.cuh"

namespace lbm {
LBM_INSTANTIATE_AA(LBM_F16S)
}  // namespace lbm
