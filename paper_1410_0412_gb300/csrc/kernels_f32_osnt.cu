// OS-NT steps for single grids.
#include "kernels.cuh"

namespace lbm {
LBM_INSTANTIATE_OSNT(LBM_F32)
}  // namespace lbm
