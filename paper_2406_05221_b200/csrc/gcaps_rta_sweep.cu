// gcaps_rta_sweep.cu -- the kernels that analyse every taskset several times in one pass
// (gcaps_rta_sweep_batch, gcaps_rta_multi_batch) and their launcher.
#include "rta_device.cuh"

using namespace gcaps_detail;

namespace {

// The same launches for a fused sweep: every taskset is read once and analysed under all the
// (timeslice, overhead) pairs of `sw`.
template <int MASK>
__global__ void __launch_bounds__(kBlockThreads, min_blocks(3))
rta_small_sweep_kernel(KParams p, const __grid_constant__ SweepArgs sw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  let_dependents_start();  // the kernel of the next size bin shares no data with this one
  u32 *warp_buf = reinterpret_cast<u32 *>(smem_raw) + (threadIdx.x >> 5) * kSmallWarpWords;
  Ahead *ahead = reinterpret_cast<Ahead *>(warp_buf + kSmallWarpWords - kAheadWords);
  run_bin<16, 2, MASK, true>(p, 3, warp_buf, ahead, &sw);
  run_bin<8, 3, MASK, true>(p, 2, warp_buf, ahead, &sw);
  run_bin<8, 2, MASK, true>(p, 1, warp_buf, ahead, &sw);
  run_bin<8, 1, MASK, true>(p, 0, warp_buf, ahead, &sw);
  wait_for_previous_grid();
}

template <int SLOTS, int MASK>
__global__ void __launch_bounds__(kBlockThreads, min_blocks(SLOTS))
rta_big_sweep_kernel(KParams p, int bin, const __grid_constant__ SweepArgs sw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  let_dependents_start();  // the kernel of the next size bin shares no data with this one
  constexpr int kWarpWords = bin_warp_words<32, SLOTS>() + kAheadWords;
  u32 *warp_buf = reinterpret_cast<u32 *>(smem_raw) + (threadIdx.x >> 5) * kWarpWords;
  Ahead *ahead = reinterpret_cast<Ahead *>(warp_buf + kWarpWords - kAheadWords);
  run_bin<32, SLOTS, MASK, true>(p, bin, warp_buf, ahead, &sw);
  wait_for_previous_grid();
}

template <int SLOTS, int MASK>
cudaError_t launch_big_sweep(const KParams &p, const SweepArgs &sw, int bin, int sm_count, cudaStream_t st) {
  constexpr int kWarps = kBlockThreads / 32;
  static int blocks_per_sm[64] = {0};
  const size_t smem = sizeof(u32) * (bin_warp_words<32, SLOTS>() + kAheadWords) * kWarps;
  return launch_persistent_ex(true, rta_big_sweep_kernel<SLOTS, MASK>, blocks_per_sm, smem,
                           (p.n_tasksets + kWarps - 1) / kWarps, sm_count, st, p, bin, sw);
}

template <int MASK>
cudaError_t launch_all_bins_sweep(const KParams &p, const SweepArgs &sw, int sm_count, cudaStream_t st) {
  constexpr int kWarps = kBlockThreads / 32;
  static int blocks_per_sm[64] = {0};
  const size_t smem = sizeof(u32) * kSmallWarpWords * kWarps;
  cudaError_t e = launch_persistent(rta_small_sweep_kernel<MASK>, blocks_per_sm, smem,
                                    (p.n_tasksets + kWarps - 1) / kWarps, sm_count, st, p, sw);
  if (e == cudaSuccess) e = launch_big_sweep<2, MASK>(p, sw, 4, sm_count, st);
  if (e == cudaSuccess) e = launch_big_sweep<3, MASK>(p, sw, 5, sm_count, st);
  if (e == cudaSuccess) e = launch_big_sweep<4, MASK>(p, sw, 6, sm_count, st);
  if (e == cudaSuccess) e = launch_big_sweep<6, MASK>(p, sw, 7, sm_count, st);
  if (e == cudaSuccess) e = launch_big_sweep<8, MASK>(p, sw, 8, sm_count, st);
  return e;
}

}  // namespace

namespace gcaps_detail {

cudaError_t launch_sweep_set(const KParams &p, const SweepArgs &sw, int sm_count, cudaStream_t st) {
  switch (sw.enabled) {
    case 1: return launch_all_bins_sweep<1>(p, sw, sm_count, st);
    case 2: return launch_all_bins_sweep<2>(p, sw, sm_count, st);
    case 4: return launch_all_bins_sweep<4>(p, sw, sm_count, st);
    case 8: return launch_all_bins_sweep<8>(p, sw, sm_count, st);
    case 5: return launch_all_bins_sweep<5>(p, sw, sm_count, st);   // GCAPS + RR, self-suspension
    case 10: return launch_all_bins_sweep<10>(p, sw, sm_count, st);  // GCAPS + RR, busy-waiting
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace gcaps_detail
