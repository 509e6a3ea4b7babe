// Two-exchange complex64 pair-convolution kernel of the 16^3 grid.
#include "launch.cuh"
#include "pairconv_wide.cuh"

namespace hse {

cudaError_t launch_pairconv_wide16(const PairArgs& args, cudaStream_t stream) {
  static bool attr_done[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!attr_done[dev]) {
    const cudaError_t err = cudaFuncSetAttribute(pairconv_wide16_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)Wide16::SMEM_REQUEST);
    if (err != cudaSuccess) return err;
    attr_done[dev] = true;
  }
  CUtensorMap tmap;
  const cudaError_t err = make_partner_tmap(&tmap, args.part, 16, (long long)args.nk_part * args.n_part * 256, 16, 256, true);
  if (err != cudaSuccess) return err;
  const unsigned grid = (unsigned)((size_t)args.nsplit * args.nk_own * args.ntiles);
  pairconv_wide16_kernel<<<grid, Wide16::THREADS, Wide16::SMEM_REQUEST, stream>>>(args, tmap);
  count_launch();
  return cudaGetLastError();
}

}  // namespace hse
