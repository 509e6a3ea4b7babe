// Two-exchange complex64 pair-convolution kernel of the 16^3 grid.
#include "launch.cuh"
#include "pairconv_wide.cuh"

namespace hse {

namespace {

template <class K>
cudaError_t set_wide_smem(K kernel, bool (&done)[64]) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!done[dev]) {
    const cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Wide16::SMEM_REQUEST);
    if (err != cudaSuccess) return err;
    done[dev] = true;
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_pairconv_wide16(int mode, const PairArgs& args, cudaStream_t stream) {
  static bool done_apply[64] = {}, done_occ[64] = {}, done_occ_w[64] = {};
  const long long rows = (long long)args.nk_part * args.n_part * 256;
  CUtensorMap tmap, tmap2;
  cudaError_t err = make_partner_tmap(&tmap, args.part, 16, rows, 16, 256, true);
  if (err != cudaSuccess) return err;
  const unsigned grid = args.item_count > 0 ? (unsigned)args.item_count
                                            : (unsigned)((size_t)args.nsplit * args.nk_own * args.ntiles);
  if (mode == MODE_APPLY) {
    err = set_wide_smem(pairconv_wide16_kernel, done_apply);
    if (err != cudaSuccess) return err;
    pairconv_wide16_kernel<<<grid, Wide16::THREADS, Wide16::SMEM_REQUEST, stream>>>(args, tmap);
  } else {
    err = make_partner_tmap(&tmap2, args.part2, 16, rows, 16, 256, true);
    if (err == cudaSuccess) err = set_wide_smem(pairconv_wide16_occ_kernel<false>, done_occ);
    if (err == cudaSuccess) err = set_wide_smem(pairconv_wide16_occ_kernel<true>, done_occ_w);
    if (err != cudaSuccess) return err;
    if (args.vtab2)
      pairconv_wide16_occ_kernel<true><<<grid, Wide16::THREADS, Wide16::SMEM_REQUEST, stream>>>(args, tmap, tmap2);
    else
      pairconv_wide16_occ_kernel<false><<<grid, Wide16::THREADS, Wide16::SMEM_REQUEST, stream>>>(args, tmap, tmap2);
  }
  count_launch();
  return cudaGetLastError();
}

}  // namespace hse
