// Split-precision tensor-core product instances for one kernel family (see kmv_x3.cuh).
#include "kmv_x3.cuh"

namespace ap {
cudaError_t launch_x3_m32(const KmvParams& p, int D, int C, cudaStream_t st) {
    return x3::dispatch<AP_MATERN32>(p, D, C, st);
}
}  // namespace ap
