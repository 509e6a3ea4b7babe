// Fused FP64 pair convolutions, axes up to 12.
#include "fused_f64_launch.cuh"

namespace hse {
cudaError_t launch_fused_f64_12(const F64Args& a, cudaStream_t stream) { return launch_fused_f64_n<12>(a, stream); }
}  // namespace hse
