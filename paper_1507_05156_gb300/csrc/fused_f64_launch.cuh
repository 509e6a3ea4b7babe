// fused_f64_launch.cuh - launch of one instantiation of the fused FP64 kernel.
#pragma once

#include <algorithm>

#include "fused_f64.cuh"
#include "launch.cuh"

namespace hse {

template <int LMAX>
cudaError_t launch_fused_f64_n(const F64Args& a, cudaStream_t stream) {
  static bool attr_done[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!attr_done[dev]) {
    const cudaError_t err =
        cudaFuncSetAttribute(fused_f64_kernel<LMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, kF64MaxSmem);
    if (err != cudaSuccess) return err;
    attr_done[dev] = true;
  }
  const int threads = f64_cta_threads(a.n1, a.n2, a.n3, a.T);
  const size_t items = (size_t)a.nsplit * a.ntiles * (a.mode == F64_ENERGY ? 1 : a.nk_own);
  fused_f64_kernel<LMAX><<<(unsigned)items, threads, a.T * f64_grid_bytes(a.n1, a.n2, a.n3), stream>>>(a);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_fused_f64_12(const F64Args& a, cudaStream_t stream);
cudaError_t launch_fused_f64_16(const F64Args& a, cudaStream_t stream);
cudaError_t launch_fused_f64_24(const F64Args& a, cudaStream_t stream);
cudaError_t launch_fused_f64_32(const F64Args& a, cudaStream_t stream);

}  // namespace hse
