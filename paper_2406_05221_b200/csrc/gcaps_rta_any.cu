// gcaps_rta_any.cu -- the kernels that walk all nine size bins in one launch (batches of at most
// 8,192 tasksets) and their launcher.  (A translation unit of its own: it holds one copy of the
// device code per size bin and analysis, and compiling it beside the others shortens the build.)
#include "rta_device.cuh"

using namespace gcaps_detail;

namespace {

// All nine bins in one launch, for batches so small (at most kPlanSmall tasksets) that the
// launches of a call cost more than its work: a call is then the one-block plan kernel and this.
// Registers and shared memory are those of the largest bin, which such a batch can afford.
constexpr int kAnyWarpWords = cmax(kSmallWarpWords, bin_warp_words<32, 8>() + kAheadWords);
template <int MODE>
__global__ void __launch_bounds__(kBlockThreads, 2) rta_any_kernel(KParams p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  let_dependents_start();
  u32 *warp_buf = reinterpret_cast<u32 *>(smem_raw) + (threadIdx.x >> 5) * kAnyWarpWords;
  Ahead *ahead = reinterpret_cast<Ahead *>(warp_buf + kAnyWarpWords - kAheadWords);
  run_bin<32, 8, 1 << MODE>(p, 8, warp_buf, ahead);
  run_bin<32, 6, 1 << MODE>(p, 7, warp_buf, ahead);
  run_bin<32, 4, 1 << MODE>(p, 6, warp_buf, ahead);
  run_bin<32, 3, 1 << MODE>(p, 5, warp_buf, ahead);
  run_bin<32, 2, 1 << MODE>(p, 4, warp_buf, ahead);
  run_bin<16, 2, 1 << MODE>(p, 3, warp_buf, ahead);
  run_bin<8, 3, 1 << MODE>(p, 2, warp_buf, ahead);
  run_bin<8, 2, 1 << MODE>(p, 1, warp_buf, ahead);
  run_bin<8, 1, 1 << MODE>(p, 0, warp_buf, ahead);
  wait_for_previous_grid();
}

}  // namespace

namespace gcaps_detail {

cudaError_t launch_any_bins(int mode, const KParams &p, int sm_count, cudaStream_t st) {
  constexpr int kWarps = kBlockThreads / 32;
  static int blocks_per_sm[4][64] = {{0}};
  const size_t smem = sizeof(u32) * kAnyWarpWords * kWarps;
  const long long want = (p.n_tasksets + kWarps - 1) / kWarps;
  switch (mode) {
    case 0: return launch_persistent(rta_any_kernel<0>, blocks_per_sm[0], smem, want, sm_count, st, p);
    case 1: return launch_persistent(rta_any_kernel<1>, blocks_per_sm[1], smem, want, sm_count, st, p);
    case 2: return launch_persistent(rta_any_kernel<2>, blocks_per_sm[2], smem, want, sm_count, st, p);
    case 3: return launch_persistent(rta_any_kernel<3>, blocks_per_sm[3], smem, want, sm_count, st, p);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace gcaps_detail
