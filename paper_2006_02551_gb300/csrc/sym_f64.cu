// The symmetric CUDA-core stage in FP64.
#include "sym_kernels.cuh"

namespace wadg {
WADG_SYM_INSTANTIATE(double)
}  // namespace wadg
