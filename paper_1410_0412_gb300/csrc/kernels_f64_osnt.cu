// OS-NT steps for IEEE double grids.
#include "kernels.cuh"

namespace lbm {
LBM_INSTANTIATE_OSNT(LBM_F64)
}  // namespace lbm
