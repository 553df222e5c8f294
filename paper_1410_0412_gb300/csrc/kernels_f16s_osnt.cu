// OS-NT steps for shifted FP16 grids.
#include "kernels.cuh"

namespace lbm {
LBM_INSTANTIATE_OSNT(LBM_F16S)
}  // namespace lbm
