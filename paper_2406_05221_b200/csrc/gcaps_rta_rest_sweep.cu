// gcaps_rta_rest_sweep.cu -- several analyses of what lies behind tiles in the stream (run_rest of rta_device.cuh).
#include "rta_device.cuh"

using namespace gcaps_detail;

namespace {

template <bool LARGE, int MASK>
__global__ void __launch_bounds__(kBlockThreads, min_blocks(LARGE ? 6 : 3))
rta_rest_sweep_kernel(KParams p, const __grid_constant__ SweepArgs sw) {
  run_rest<LARGE, MASK, true>(p, &sw);
}

template <int MASK>
cudaError_t launch_both(const KParams &p, const SweepArgs &sw, int sm_count, cudaStream_t st) {
  static int small_blocks[64] = {0}, large_blocks[64] = {0};
  const cudaError_t e = launch_rest_part<false>(rta_rest_sweep_kernel<false, MASK>, small_blocks, sm_count, st, p, sw);
  return e == cudaSuccess ? launch_rest_part<true>(rta_rest_sweep_kernel<true, MASK>, large_blocks, sm_count, st, p, sw) : e;
}

}  // namespace

namespace gcaps_detail {

cudaError_t launch_sweep_rest(const KParams &p, const SweepArgs &sw, int sm_count, cudaStream_t st) {
  switch (sw.enabled) {
    case 1: return launch_both<1>(p, sw, sm_count, st);
    case 2: return launch_both<2>(p, sw, sm_count, st);
    case 4: return launch_both<4>(p, sw, sm_count, st);
    case 8: return launch_both<8>(p, sw, sm_count, st);
    case 5: return launch_both<5>(p, sw, sm_count, st);   // GCAPS + RR, self-suspension
    case 10: return launch_both<10>(p, sw, sm_count, st);  // GCAPS + RR, busy-waiting
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace gcaps_detail
