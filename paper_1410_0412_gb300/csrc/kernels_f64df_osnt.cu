// OS-NT steps for double-float arithmetic on IEEE double grids.
#include "kernels.cuh"

namespace lbm {
LBM_INSTANTIATE_OSNT(LBM_F64_DF)
}  // namespace lbm
