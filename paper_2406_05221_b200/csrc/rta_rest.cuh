// rta_rest.cuh -- what lies behind tiles in the stream: the tasksets that these listed as left over, or all size bins where the
// batch was none for tiles.  Internal.
#ifndef GCAPS_RTA_REST_CUH_
#define GCAPS_RTA_REST_CUH_

#include "rta_device.cuh"

namespace {

// Two launches share the bins: up to 96 tasks, and larger tasksets, which need twice the registers.  The first one is launched while
// the one in front of it is under way and waits for that; its blocks let the second go only then, so that it finds the header complete.  (A
// launch that finds nothing to do costs a call 1.7 us; one per bin, as behind a plan, would be six more.)
template <bool LARGE>
__host__ __device__ constexpr int rest_warp_words() {
  return LARGE ? bin_warp_words<32, 8>() + kAheadWords : cmax(kSmallWarpWords, bin_warp_words<32, 3>() + kAheadWords);
}
template <bool LARGE, int MASK, bool SWEEP>
__device__ __forceinline__ void run_rest(const KParams &p, const SweepArgs *sw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (!LARGE) wait_for_previous_grid();
  let_dependents_start();
  // (one look at all counts: mostly there is nothing to do)
  const int lane = threadIdx.x & 31;
  const bool any = __any_sync(kFull, lane >= (LARGE ? 6 : 0) && lane < (LARGE ? kNumBins : 6) && p.hdr->bin_count[lane < kNumBins ? lane : 0] > 0);
  if (!any) {
    if (LARGE) wait_for_previous_grid();
    return;
  }
  u32 *const buf = reinterpret_cast<u32 *>(smem_raw) + (threadIdx.x >> 5) * rest_warp_words<LARGE>();
  Ahead *const ahead = reinterpret_cast<Ahead *>(buf + rest_warp_words<LARGE>() - kAheadWords);
  if constexpr (LARGE) {
    run_bin<32, 8, MASK, SWEEP>(p, 8, buf, ahead, sw);
    run_bin<32, 6, MASK, SWEEP>(p, 7, buf, ahead, sw);
    run_bin<32, 4, MASK, SWEEP>(p, 6, buf, ahead, sw);
    wait_for_previous_grid();
  } else {
    run_bin<32, 3, MASK, SWEEP>(p, 5, buf, ahead, sw);
    run_bin<32, 2, MASK, SWEEP>(p, 4, buf, ahead, sw);
    run_bin<16, 2, MASK, SWEEP>(p, 3, buf, ahead, sw);
    run_bin<8, 3, MASK, SWEEP>(p, 2, buf, ahead, sw);
    run_bin<8, 2, MASK, SWEEP>(p, 1, buf, ahead, sw);
    run_bin<8, 1, MASK, SWEEP>(p, 0, buf, ahead, sw);
  }
}

// As launch_persistent_ex; `kernel` calls run_rest.
template <bool LARGE, typename... Args>
cudaError_t launch_rest_part(void (*kernel)(KParams, Args...), int *blocks_per_sm, int sm_count, cudaStream_t st, const KParams &p,
                             Args... args) {
  constexpr int kWarps = kBlockThreads / 32;
  return launch_persistent_ex(true, kernel, blocks_per_sm, sizeof(u32) * rest_warp_words<LARGE>() * kWarps,
                              (p.n_tasksets + kWarps - 1) / kWarps, sm_count, st, p, args...);
}

}  // namespace
#endif  // GCAPS_RTA_REST_CUH_
