// Fused FP64 pair convolutions, an axis longer than 24.
#include "fused_f64_launch.cuh"

namespace hse {
cudaError_t launch_fused_f64_32(const F64Args& a, cudaStream_t stream) { return launch_fused_f64_n<32>(a, stream); }
}  // namespace hse
