// gcaps_rta_direct_sweep.cu -- several analyses of a batch of at most kDirectSweepMost tasksets in one launch, a
// block of one warp per taskset and share of the pairs, no plan.
#include "rta_device.cuh"

using namespace gcaps_detail;

namespace {

constexpr int kDirectWords = bin_warp_words<32, 8>();

// Block (t, y) stages taskset t and takes the y-th share of the (timeslice, overhead) pairs: as long as the
// batch does not fill the device, staging a taskset several times costs nothing and the pairs run side by
// side (10 pairs under GCAPS of 1,000 20-task tasksets: 70 us, 81 us unshared; 172 us with plan and binned
// kernels).  4,000 tasksets take 79 to 202 us here and 80 to 278 us there; 8,192 tasksets up to 346
// against 258 us.
template <int MASK>
__global__ void __launch_bounds__(32) rta_direct_sweep_kernel(KParams p, const __grid_constant__ SweepArgs sw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  u32 *const buf = reinterpret_cast<u32 *>(smem_raw);
  const int lane = threadIdx.x;
  const i64 t = blockIdx.x;
  const int q0 = (int)(blockIdx.y * sw.n / gridDim.y), q1 = (int)((blockIdx.y + 1) * sw.n / gridDim.y);
  const i64 a = p.task_off[t] - p.task_base, b = p.task_off[t + 1] - p.task_base;
  int how = kFastDeclined;
  if (a >= 0 && b > a && b <= p.n_tasks && b - a <= GCAPS_RTA_MAX_TASKS && sw.max_ovh < (1 << 20)) {
    const int n = (int)(b - a);
    if (n <= 32) how = analyse_fast<32, 1, MASK, true, true>(p, true, t, a, n, buf, lane, kFull, &sw, q0, q1);
    else if (n <= 64) how = analyse_fast<32, 2, MASK, true, true>(p, true, t, a, n, buf, lane, kFull, &sw, q0, q1);
    else if (n <= 96) how = analyse_fast<32, 3, MASK, true, true>(p, true, t, a, n, buf, lane, kFull, &sw, q0, q1);
    else if (n <= 128) how = analyse_fast<32, 4, MASK, true, true>(p, true, t, a, n, buf, lane, kFull, &sw, q0, q1);
    else if (n <= 192) how = analyse_fast<32, 6, MASK, true, true>(p, true, t, a, n, buf, lane, kFull, &sw, q0, q1);
    else how = analyse_fast<32, 8, MASK, true, true>(p, true, t, a, n, buf, lane, kFull, &sw, q0, q1);
  }
  __syncwarp();
  if (how != kFastDone)
    exact_by_pair<32, 256, MASK>(p, sw, t, *reinterpret_cast<GroupSmem<256> *>(buf), lane, kFull, q0, q1);
}

template <int MASK>
cudaError_t launch_direct_sweep(const KParams &p, const SweepArgs &sw, int sm_count, cudaStream_t st) {
  constexpr int smem = (int)(sizeof(u32) * kDirectWords);
  static_assert(sizeof(GroupSmem<256>) <= (size_t)smem && smem <= 48 * 1024, "no attribute to set");
  long long shares = 16LL * sm_count / p.n_tasksets;
  shares = shares < 1 ? 1 : shares > sw.n ? sw.n : shares;
  rta_direct_sweep_kernel<MASK><<<dim3((unsigned int)p.n_tasksets, (unsigned int)shares), 32, smem, st>>>(p, sw);
  return cudaGetLastError();
}

}  // namespace

namespace gcaps_detail {

cudaError_t launch_sweep_one_warp_each(const KParams &p, const SweepArgs &sw, int sm_count, cudaStream_t st) {
  switch (sw.enabled) {
    case 1: return launch_direct_sweep<1>(p, sw, sm_count, st);
    case 2: return launch_direct_sweep<2>(p, sw, sm_count, st);
    case 4: return launch_direct_sweep<4>(p, sw, sm_count, st);
    case 8: return launch_direct_sweep<8>(p, sw, sm_count, st);
    case 5: return launch_direct_sweep<5>(p, sw, sm_count, st);
    case 10: return launch_direct_sweep<10>(p, sw, sm_count, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace gcaps_detail
