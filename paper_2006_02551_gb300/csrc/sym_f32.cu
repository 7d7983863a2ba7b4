// The symmetric CUDA-core stage in FP32.
#include "sym_kernels.cuh"

namespace wadg {
WADG_SYM_INSTANTIATE(float)
}  // namespace wadg
