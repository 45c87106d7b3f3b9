// gcaps_rta_direct.cu -- the kernels of batches of at most kDirectMost tasksets and their launcher: one
// launch, a block of one warp per taskset, no plan.  (A translation unit of its own: it holds one copy
// of the device code per size class and analysis, and compiling it beside the others shortens the
// build.)
#include "rta_device.cuh"

using namespace gcaps_detail;

namespace {

// A block of one warp per taskset, in the order of the batch.  A small batch is bound by launches and by
// one taskset's chain of dependent loads: without the plan (a launch, and two loads in front of every
// taskset) 1,184 tasksets of 8 / 20 / 80 tasks take 9 / 12 / 10 us of a stream's time under GCAPS, with
// plan and one kernel over all size bins 17 / 29 / 19 us.  It stays ahead of the binned kernels while
// these cannot fill the device.  12,288 tasksets of 8 / 20 / 80 / 128 / 192 tasks take 35 / 68 / 52 / 64 / 589 us
// under GCAPS and 39 / 31 / 55 / 68 / 70 us under RR against 44 / 66 / 79 / 92 / 876 and 45 / 50 / 76 / 91 / 102 us
// with a plan (busy-waiting modes within 10 % of these); 24,000 of 8 / 20 / 80 tasks 66 / 127 / 90 against
// 49 / 85 / 90 us.  A mixture of 4 to 192 tasks: 95 against 120 us under GCAPS, but 114 against 91 us under RR.
// (Shared memory is set aside for 256 tasks, which leaves 13 warps per SM.)  Since lanes add up their own tasks'
// segments 12,288 of 8 / 20 / 80 tasks take 31 / 63 / 47 us under GCAPS and 33 / 27 / 49 us under RR, a mixture 73 and
// 88 us; with a plan 13,000 of the mixture 119 and 92 us.
constexpr int kDirectWords = bin_warp_words<32, 8>();
template <int SLOTS, int MODE>
__device__ __forceinline__ int direct_pass(const KParams &p, i64 t, i64 a, int n, u32 *buf, int lane) {
  return analyse_fast<32, SLOTS, 1 << MODE, false, true>(p, true, t, a, n, buf, lane, kFull);
}
template <int MODE>
__global__ void __launch_bounds__(32) rta_direct_kernel(KParams p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  u32 *const buf = reinterpret_cast<u32 *>(smem_raw);
  const int lane = threadIdx.x;
  const i64 t = blockIdx.x;
  const i64 a = p.task_off[t] - p.task_base, b = p.task_off[t + 1] - p.task_base;
  int how = kFastDeclined;
  if (a >= 0 && b > a && b <= p.n_tasks && b - a <= GCAPS_RTA_MAX_TASKS && p.ovh < (1 << 20)) {
    const int n = (int)(b - a);
    if (n <= 32) how = direct_pass<1, MODE>(p, t, a, n, buf, lane);
    else if (n <= 64) how = direct_pass<2, MODE>(p, t, a, n, buf, lane);
    else if (n <= 96) how = direct_pass<3, MODE>(p, t, a, n, buf, lane);
    else if (n <= 128) how = direct_pass<4, MODE>(p, t, a, n, buf, lane);
    else if (n <= 192) how = direct_pass<6, MODE>(p, t, a, n, buf, lane);
    else how = direct_pass<8, MODE>(p, t, a, n, buf, lane);
  }
  __syncwarp();
  if (how != kFastDone)  // the exact path reads task_off again and validates everything itself
    analyse_taskset<32, 256>(p, t, *reinterpret_cast<GroupSmem<256> *>(buf), lane, kFull);
}

template <int MODE>
cudaError_t launch_direct(const KParams &p, cudaStream_t st) {
  constexpr int smem = (int)(sizeof(u32) * kDirectWords);
  static_assert(sizeof(GroupSmem<256>) <= (size_t)smem && smem <= 48 * 1024, "no attribute to set");
  rta_direct_kernel<MODE><<<(unsigned int)p.n_tasksets, 32, smem, st>>>(p);
  return cudaGetLastError();
}

}  // namespace

namespace gcaps_detail {

cudaError_t launch_one_warp_each(int mode, const KParams &p, cudaStream_t st) {
  switch (mode) {
    case 0: return launch_direct<0>(p, st);
    case 1: return launch_direct<1>(p, st);
    case 2: return launch_direct<2>(p, st);
    case 3: return launch_direct<3>(p, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace gcaps_detail
