// gcaps_rta_rest.cu -- one analysis of what lies behind tiles in the stream (run_rest of rta_device.cuh).
#include "rta_device.cuh"

using namespace gcaps_detail;

namespace {

template <bool LARGE, int MODE>
__global__ void __launch_bounds__(kBlockThreads, min_blocks(LARGE ? 6 : 3)) rta_rest_kernel(KParams p) {
  run_rest<LARGE, 1 << MODE, false>(p, nullptr);
}

template <int MODE>
cudaError_t launch_both(const KParams &p, int sm_count, cudaStream_t st) {
  static int small_blocks[64] = {0}, large_blocks[64] = {0};
  const cudaError_t e = launch_rest_part<false>(rta_rest_kernel<false, MODE>, small_blocks, sm_count, st, p);
  return e == cudaSuccess ? launch_rest_part<true>(rta_rest_kernel<true, MODE>, large_blocks, sm_count, st, p) : e;
}

}  // namespace

namespace gcaps_detail {

cudaError_t launch_rest(int mode, const KParams &p, int sm_count, cudaStream_t st) {
  switch (mode) {
    case 0: return launch_both<0>(p, sm_count, st);
    case 1: return launch_both<1>(p, sm_count, st);
    case 2: return launch_both<2>(p, sm_count, st);
    case 3: return launch_both<3>(p, sm_count, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace gcaps_detail
