// Fused FP64 pair convolutions, axes up to 16.
#include "fused_f64_launch.cuh"

namespace hse {
cudaError_t launch_fused_f64_16(const F64Args& a, cudaStream_t stream) { return launch_fused_f64_n<16>(a, stream); }

cudaError_t launch_fused_f64(const F64Args& a, cudaStream_t stream) {
  const int longest = std::max(a.n1, std::max(a.n2, a.n3));
  if (longest <= 12) return launch_fused_f64_12(a, stream);
  if (longest <= 16) return launch_fused_f64_16(a, stream);
  return longest <= 24 ? launch_fused_f64_24(a, stream) : launch_fused_f64_32(a, stream);
}
}  // namespace hse
