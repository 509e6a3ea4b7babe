// Fused FP64 pair convolutions, axes up to 24.
#include "fused_f64_launch.cuh"

namespace hse {
cudaError_t launch_fused_f64_24(const F64Args& a, cudaStream_t stream) { return launch_fused_f64_n<24>(a, stream); }
}  // namespace hse
