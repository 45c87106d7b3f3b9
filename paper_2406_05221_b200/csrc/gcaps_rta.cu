// gcaps_rta.cu -- batched worst-case response-time analysis of GPU-using real-time tasksets
// (GCAPS, ECRTS 2024, arXiv 2406.05221, Sec. 6) for NVIDIA B200 (sm_100a).
//
// This file: the plan (size binning), the kernels of a single analysis, the host side and the entry
// points.  The device code of the analysis is rta_device.cuh.
//
// Everything is integer arithmetic on microseconds.  No tensor cores: nothing here is a dense
// contraction.  No host synchronisation and no allocation in gcaps_rta_batch.
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <mutex>

#include "rta_device.cuh"
#include "rta_staged.cuh"
#include "rta_tile_kept.cuh"

using namespace gcaps_detail;

namespace {

// ---------------------------------------------------------------------------------------------
// plan: counting sort of taskset indices by size bin (histogram per block, scan, scatter)
// ---------------------------------------------------------------------------------------------
__global__ void plan_count_kernel(KParams p) {
  __shared__ unsigned int cnt[kBinStride];
  if (threadIdx.x < kBinStride) cnt[threadIdx.x] = 0;
  __syncthreads();
  i64 t0 = (i64)blockIdx.x * kPlanItems;
  for (int k = threadIdx.x; k < kPlanItems; k += blockDim.x) {
    i64 t = t0 + k;
    if (t < p.n_tasksets) atomicAdd(&cnt[size_bin(p.task_off[t + 1] - p.task_off[t])], 1u);
  }
  __syncthreads();
  if (threadIdx.x < kBinStride)
    p.block_cnt[(size_t)blockIdx.x * kBinStride + threadIdx.x] = cnt[threadIdx.x];
}

// One block, one warp per bin.  Turns per-block counts into per-block write cursors and fills the
// header.
__global__ void plan_scan_kernel(KParams p, unsigned int n_blocks) {
  __shared__ unsigned int bin_total[kBinStride];
  const int lane = threadIdx.x & 31, b = threadIdx.x >> 5;
  if (b < kNumBins) {
    unsigned int carry = 0;
    for (unsigned int base = 0; base < n_blocks; base += 32) {
      const unsigned int i = base + lane;
      const unsigned int v = i < n_blocks ? p.block_cnt[(size_t)i * kBinStride + b] : 0u;
      unsigned int x = v;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const unsigned int y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
      }
      if (i < n_blocks) p.block_cnt[(size_t)i * kBinStride + b] = carry + x - v;  // cursor within the bin
      carry += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) bin_total[b] = carry;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned int s = 0;
    for (int k = 0; k < kBinStride; ++k) {
      const unsigned int c = k < kNumBins ? bin_total[k] : 0u;
      p.hdr->bin_start[k] = s;
      p.hdr->bin_count[k] = c;
      p.hdr->next[k] = 0;
      if (k < kNumBins) p.hdr->next2[k] = 0, p.hdr->deferred[k] = 0, p.hdr->first_tries[k] = 0;
      s += c;
    }
  }
}

__global__ void plan_scatter_kernel(KParams p) {
  __shared__ unsigned int cursor[kBinStride];
  if (threadIdx.x < kBinStride)
    cursor[threadIdx.x] = p.block_cnt[(size_t)blockIdx.x * kBinStride + threadIdx.x];
  __syncthreads();
  i64 t0 = (i64)blockIdx.x * kPlanItems;
  for (int k = threadIdx.x; k < kPlanItems; k += blockDim.x) {
    i64 t = t0 + k;
    if (t < p.n_tasksets) {
      int b = size_bin(p.task_off[t + 1] - p.task_off[t]);
      unsigned int slot = atomicAdd(&cursor[b], 1u);
      p.perm[p.hdr->bin_start[b] + slot] = (unsigned int)t;
    }
  }
}

// The three steps in one block, for batches small enough that launches cost more than the work.
__global__ void __launch_bounds__(1024) plan_small_kernel(KParams p) {
  __shared__ unsigned int cnt[kBinStride], start[kBinStride];
  if (threadIdx.x < kBinStride) cnt[threadIdx.x] = 0;
  __syncthreads();
  for (i64 t = threadIdx.x; t < p.n_tasksets; t += blockDim.x)
    atomicAdd(&cnt[size_bin(p.task_off[t + 1] - p.task_off[t])], 1u);
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned int s = 0;
    for (int k = 0; k < kBinStride; ++k) {
      const unsigned int c = k < kNumBins ? cnt[k] : 0u;
      p.hdr->bin_start[k] = s;
      p.hdr->bin_count[k] = c;
      p.hdr->next[k] = 0;
      if (k < kNumBins) p.hdr->next2[k] = 0, p.hdr->deferred[k] = 0, p.hdr->first_tries[k] = 0;
      start[k] = s;
      cnt[k] = 0;  // from here on the write cursor of the bin
      s += c;
    }
  }
  __syncthreads();
  for (i64 t = threadIdx.x; t < p.n_tasksets; t += blockDim.x) {
    const int b = size_bin(p.task_off[t + 1] - p.task_off[t]);
    p.perm[start[b] + atomicAdd(&cnt[b], 1u)] = (unsigned int)t;
  }
}

// Behind tiles: where the batch was none for them they have counted its size bins, and this is the rest of the plan.  Blocks of
// tasksets get their places in the permutation from a counter per bin.
__global__ void __launch_bounds__(256) plan_behind_tiles_kernel(KParams p) {
  __shared__ unsigned int cnt[kBinStride], cursor[kBinStride];
  wait_for_previous_grid();
  let_dependents_start();
  if (p.hdr->in_tiles) return;
  const int bin = threadIdx.x;
  unsigned int start = 0;
  if (bin < kNumBins) {
    for (int k = 0; k < bin; ++k) start += p.hdr->bin_count[k];
    if (blockIdx.x == 0) p.hdr->bin_start[bin] = start;
  }
#pragma unroll 1
  for (i64 t0 = (i64)blockIdx.x * kPlanItems; t0 < p.n_tasksets; t0 += (i64)gridDim.x * kPlanItems) {
    if (bin < kNumBins) cnt[bin] = 0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kPlanItems; k += 256) {
      const i64 t = t0 + k + threadIdx.x;
      if (t < p.n_tasksets) atomicAdd(&cnt[size_bin(p.task_off[t + 1] - p.task_off[t])], 1u);
    }
    __syncthreads();
    if (bin < kNumBins) cursor[bin] = start + atomicAdd(&p.hdr->next2[bin], cnt[bin]);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kPlanItems; k += 256) {
      const i64 t = t0 + k + threadIdx.x;
      if (t < p.n_tasksets) p.perm[atomicAdd(&cursor[size_bin(p.task_off[t + 1] - p.task_off[t])], 1u)] = (unsigned int)t;
    }
    __syncthreads();
  }
}

// The bins of up to 32 tasks in one persistent launch, largest tasksets first: (lanes per
// taskset, tasks per lane) = (16,2) (8,3) (8,2) (8,1) for at most 32, 24, 16, 8 tasks, i.e. two or
// four tasksets per warp.  (A look at the first ranks out of a stage, a warp per taskset, was slower
// here in every form tried: 100,000 24-task tasksets under round robin 163 us against 128.)
template <int MODE>
__global__ void __launch_bounds__(kBlockThreads, min_blocks(3)) rta_small_kernel(KParams p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  let_dependents_start();  // the kernel of the next size bin shares no data with this one
  u32 *warp_buf = reinterpret_cast<u32 *>(smem_raw) + (threadIdx.x >> 5) * kSmallWarpWords;
  Ahead *ahead = reinterpret_cast<Ahead *>(warp_buf + kSmallWarpWords - kAheadWords);
  run_bin<16, 2, 1 << MODE>(p, 3, warp_buf, ahead);
  run_bin<8, 3, 1 << MODE>(p, 2, warp_buf, ahead);
  run_bin<8, 2, 1 << MODE>(p, 1, warp_buf, ahead);
  run_bin<8, 1, 1 << MODE>(p, 0, warp_buf, ahead);
  wait_for_previous_grid();
}

// First launch of a bin of larger tasksets: a warp per taskset, SLOTS tasks per lane.
template <int SLOTS, int MODE>
__global__ void __launch_bounds__(kStagedThreads, staged_min_blocks(SLOTS))
rta_big_kernel(KParams p, int bin, u32 stage_bytes) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ SliceTable tab;
  let_dependents_start();  // the kernel of the next size bin shares no data with this one
  if (threadIdx.x == 0) {
    tab.ptr[0] = p.period, tab.ptr[1] = p.deadline, tab.ptr[2] = p.priority, tab.ptr[3] = p.core;
    tab.ptr[4] = p.cseg_off, tab.ptr[5] = p.gseg_off;
    tab.ptr[6] = p.cseg_wcet, tab.ptr[7] = p.gseg_misc, tab.ptr[8] = p.gseg_exec;
#pragma unroll
    for (int k = 0; k < kArrays; ++k)
      tab.len[k] = k < 4 ? p.n_tasks : (k < 6 ? p.n_tasks + 1 : (k == 6 ? p.n_csegs : p.n_gsegs));
  }
  __syncthreads();
  unsigned char *mine = smem_raw + (threadIdx.x >> 5) * (sizeof(StagedWarp<SLOTS>) + stage_bytes);
  run_staged_bin<SLOTS, MODE>(p, bin, stage_bytes, *reinterpret_cast<StagedWarp<SLOTS> *>(mine),
                              mine + sizeof(StagedWarp<SLOTS>), tab);
  wait_for_previous_grid();
}

// Second launches: what the first ones marked, largest tasksets first.  LARGE: the bins of more than 96
// tasks, which need twice the registers.  The other one is launched first and waits for the marks; its blocks let
// the LARGE launch go only after that, so that one finds the marks complete as it starts and runs beside it
// (100,000 `divergence` tasksets at an overhead of 2 us 1,014 -> 890 us together with the entries being
// pulled, see run_deferred_bin).
template <bool LARGE>
__host__ __device__ constexpr int deferred_warp_words() {
  return bin_warp_words<32, LARGE ? 8 : 3>() + kAheadWords;
}
template <bool LARGE, int MODE>
__global__ void __launch_bounds__(kBlockThreads, min_blocks(LARGE ? 6 : 3)) rta_deferred_kernel(KParams p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if constexpr (!LARGE) wait_for_previous_grid();  // the marks in the permutation are complete from here on
  let_dependents_start();
  u32 *buf = reinterpret_cast<u32 *>(smem_raw) + (threadIdx.x >> 5) * deferred_warp_words<LARGE>();
  Ahead *ahead = reinterpret_cast<Ahead *>(buf + deferred_warp_words<LARGE>() - kAheadWords);
  if constexpr (LARGE) {
    run_deferred_bin<8, MODE>(p, 8, buf, ahead);
    run_deferred_bin<6, MODE>(p, 7, buf, ahead);
    run_deferred_bin<4, MODE>(p, 6, buf, ahead);
    wait_for_previous_grid();
  } else {
    run_deferred_bin<3, MODE>(p, 5, buf, ahead);
    run_deferred_bin<2, MODE>(p, 4, buf, ahead);
  }
}

// ---------------------------------------------------------------------------------------------
// validation kernel: one thread per taskset
// ---------------------------------------------------------------------------------------------
__global__ void validate_kernel(KParams p, int32_t *out_err) {
  const i64 t = (i64)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= p.n_tasksets) return;
  const i64 a = p.task_off[t], b = p.task_off[t + 1];
  if (a < 0 || b < a || b > p.n_tasks || b - a > GCAPS_RTA_MAX_TASKS) {
    out_err[t] = GCAPS_BAD_TASK_RANGE;
    return;
  }
  int bad = 0;
  for (i64 k = a; k < b; ++k) {
    const i64 c0 = p.cseg_off[k], c1 = p.cseg_off[k + 1], g0 = p.gseg_off[k], g1 = p.gseg_off[k + 1];
    const bool seg_ok = !(c0 < 0 || c1 < c0 || c1 > p.n_csegs || c1 - c0 > GCAPS_RTA_MAX_SEGMENTS ||
                          g0 < 0 || g1 < g0 || g1 > p.n_gsegs || g1 - g0 > GCAPS_RTA_MAX_SEGMENTS);
    if (!seg_ok) bad |= GCAPS_BAD_SEG_RANGE;
    const i64 T = p.period[k], D = p.deadline[k], c = p.core[k];
    if (T < 1 || T > GCAPS_RTA_MAX_TIME) bad |= GCAPS_BAD_PERIOD;
    if (D < 1 || D > T) bad |= GCAPS_BAD_DEADLINE;
    if (c < 0 || c > GCAPS_RTA_MAX_CORE) bad |= GCAPS_BAD_CORE;
    if (seg_ok) {
      for (i64 j = c0; j < c1; ++j)
        if (p.cseg_wcet[j] < 0 || p.cseg_wcet[j] > GCAPS_RTA_MAX_TIME) bad |= GCAPS_BAD_WCET;
      for (i64 j = g0; j < g1; ++j)
        if (p.gseg_misc[j] < 0 || p.gseg_misc[j] > GCAPS_RTA_MAX_TIME || p.gseg_exec[j] < 0 ||
            p.gseg_exec[j] > GCAPS_RTA_MAX_TIME)
          bad |= GCAPS_BAD_WCET;
    }
  }
  out_err[t] = bad;
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

size_t plan_blocks(int64_t n_tasksets) { return (size_t)((n_tasksets + kPlanItems - 1) / kPlanItems); }

}  // namespace


// ---------------------------------------------------------------------------------------------
// host side shared with the other translation units of the library
// ---------------------------------------------------------------------------------------------
namespace gcaps_detail {

thread_local int g_last_cuda_error = 0;
std::mutex g_init_mutex;

static DeviceInfo g_dev[64];

int device_info(DeviceInfo *out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) {
    g_last_cuda_error = (int)e;
    return GCAPS_ERR_NO_DEVICE;
  }
  if (dev < 0 || dev >= 64) return GCAPS_ERR_NO_DEVICE;
  std::lock_guard<std::mutex> lock(g_init_mutex);
  if (g_dev[dev].ok == 0) {
    int major = 0, sms = 0;
    e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) {
      g_last_cuda_error = (int)e;
      return GCAPS_ERR_NO_DEVICE;
    }
    g_dev[dev].sm_count = sms;
    g_dev[dev].ok = major == 10 ? 1 : -1;
  }
  if (g_dev[dev].ok != 1) return GCAPS_ERR_NO_DEVICE;
  *out = g_dev[dev];
  return GCAPS_OK;
}

int check_args(const gcaps_tasksets_t *ts, int64_t n_tasksets, int policy, int64_t L, int64_t ovh) {
  if (!ts || n_tasksets < 0 || n_tasksets > 0x7fffffffLL) return GCAPS_ERR_INVALID_ARG;
  const int pol = policy & 0xff;
  if (pol != GCAPS_POLICY_GCAPS && pol != GCAPS_POLICY_RR) return GCAPS_ERR_INVALID_ARG;
  if (policy & ~(0xff | GCAPS_RTA_BUSY | GCAPS_RTA_LITERAL | GCAPS_RTA_BEST_EFFORT))
    return GCAPS_ERR_INVALID_ARG;
  if (ovh < 0 || ovh > GCAPS_RTA_MAX_TIME) return GCAPS_ERR_INVALID_ARG;
  if (pol == GCAPS_POLICY_RR && (L < 1 || L > GCAPS_RTA_MAX_TIME)) return GCAPS_ERR_INVALID_ARG;
  if (ts->n_tasks < 0 || ts->n_csegs < 0 || ts->n_gsegs < 0) return GCAPS_ERR_INVALID_ARG;
  if (n_tasksets > 0) {
    if (!ts->task_off) return GCAPS_ERR_INVALID_ARG;
    if (ts->n_tasks > 0 && (!ts->period || !ts->deadline || !ts->priority || !ts->core ||
                            !ts->cseg_off || !ts->gseg_off))
      return GCAPS_ERR_INVALID_ARG;
    if (ts->n_csegs > 0 && !ts->cseg_wcet) return GCAPS_ERR_INVALID_ARG;
    if (ts->n_gsegs > 0 && (!ts->gseg_misc || !ts->gseg_exec)) return GCAPS_ERR_INVALID_ARG;
  }
  return GCAPS_OK;
}

void fill_params(KParams *p, const gcaps_tasksets_t *ts, int64_t n_tasksets, int policy, int64_t L,
                 int64_t ovh, int64_t *out_wcrt, uint8_t *out_sched) {
  memset(p, 0, sizeof(*p));
  p->task_off = (const i64 *)ts->task_off;
  p->period = (const i64 *)ts->period;
  p->deadline = (const i64 *)ts->deadline;
  p->priority = (const i64 *)ts->priority;
  p->core = (const i64 *)ts->core;
  p->cseg_off = (const i64 *)ts->cseg_off;
  p->cseg_wcet = (const i64 *)ts->cseg_wcet;
  p->gseg_off = (const i64 *)ts->gseg_off;
  p->gseg_misc = (const i64 *)ts->gseg_misc;
  p->gseg_exec = (const i64 *)ts->gseg_exec;
  p->n_tasks = ts->n_tasks;
  p->n_csegs = ts->n_csegs;
  p->n_gsegs = ts->n_gsegs;
  p->n_tasksets = n_tasksets;
  p->policy = policy;
  p->L = (policy & 0xff) == GCAPS_POLICY_RR ? L : 1;
  p->ovh = ovh;
  if (p->L == 1) {
    p->l_mode = 1;
  } else if (p->L >= (i64)kFastLimit) {
    p->l_mode = 2;
  } else {
    p->l_mode = 0;
    make_reciprocal((u32)p->L, p->l_magic, p->l_shift);
  }
  p->out_wcrt = (i64 *)out_wcrt;
  p->out_sched = out_sched;
}

int place_plan(KParams &p, void *workspace, size_t workspace_bytes) {
  const size_t need = gcaps_rta_workspace_bytes(p.n_tasksets);
  if (!workspace || workspace_bytes < need || ((uintptr_t)workspace & 255u))
    return GCAPS_ERR_WORKSPACE;
  unsigned char *w = (unsigned char *)workspace;
  const size_t nb = plan_blocks(p.n_tasksets);
  p.hdr = (PlanHeader *)w;
  p.block_cnt = (unsigned int *)(w + 256);
  p.perm = (unsigned int *)(w + 256 + align_up(nb * kBinStride * sizeof(unsigned int), 256));
  return GCAPS_OK;
}

static void enqueue_plan_kernels(const KParams &p, cudaStream_t st) {
  const size_t nb = plan_blocks(p.n_tasksets);
  if (p.n_tasksets <= kPlanSmall) {
    plan_small_kernel<<<1, 1024, 0, st>>>(p);
    return;
  }
  plan_count_kernel<<<(unsigned int)nb, 256, 0, st>>>(p);
  plan_scan_kernel<<<1, 32 * kNumBins, 0, st>>>(p, (unsigned int)nb);
  plan_scatter_kernel<<<(unsigned int)nb, 256, 0, st>>>(p);
}

int enqueue_plan(KParams &p, void *workspace, size_t workspace_bytes, cudaStream_t st) {
  const int rc = place_plan(p, workspace, workspace_bytes);
  if (rc == GCAPS_OK) enqueue_plan_kernels(p, st);
  return rc;
}

}  // namespace gcaps_detail

namespace {

// The stage of a bin: room for a taskset of the bin's largest size with a tenth more segments per task
// than the batch has on average, as long as an SM then still holds kMinStages of them.  Four hold whatever
// the 32-bit path takes.  (With eight, most tasksets of 256 tasks and of 192 with many segments did not fit
// and went to the second launch: 100,000 of 256 tasks with 1 to 5 GPU segments 1,089 -> 521 us under RR and
// 935 -> 520 us under GCAPS, 12,289 of them 385 -> 119 us.)  Where the
// batch's mean size lies in the bin its tasksets are probably alike, and 5 % above the mean (but no
// less than the middle of the bin) has to do: more stages, i.e. more warps, per SM count for more
// than the few tasksets left over (80-task tasksets: 18 instead of 16 warps, 1.53 instead of 1.64 ms
// per 1,000,000).
constexpr int kMinStages = 4;

template <int SLOTS, int MODE>
cudaError_t launch_big(const KParams &p, int bin, int sm_count, cudaStream_t st) {
  constexpr int kWarps = kStagedThreads / 32;
  constexpr size_t kFixed = sizeof(StagedWarp<SLOTS>);
  constexpr size_t kLeast = sizeof(u32) * FastLayout<32, SLOTS>::kWords;  // the full pass works in a stage too
  constexpr size_t kMost = (kSmemPerSm / kMinStages - kSmemPerBlockReserved - kFixed) / 16 * 16;
  static_assert(kFixed % 16 == 0 && kLeast <= kMost, "stages are 16-byte aligned");
  static int blocks_by_registers[64] = {0};
  const double per_task = 48.0 + 8.8 * ((double)p.n_csegs + 2.0 * (double)p.n_gsegs) / (double)(p.n_tasks > 0 ? p.n_tasks : 1);
  constexpr double kTasksLo = SLOTS <= 4 ? 32 * (SLOTS - 1) : 32 * (SLOTS - 2), kTasksHi = 32 * SLOTS;
  const double mean = (double)p.n_tasks / (double)p.n_tasksets;
  double tasks = kTasksHi;
  if (mean > kTasksLo && 1.05 * mean < kTasksHi) tasks = 1.05 * mean > (kTasksLo + kTasksHi) / 2 ? 1.05 * mean : (kTasksLo + kTasksHi) / 2;
  const double want = per_task * tasks + 9 * 24;
  size_t stage = want > (double)kMost ? kMost : ((size_t)want + 15) / 16 * 16;
  if (stage < kLeast) stage = (kLeast + 15) / 16 * 16;
  const size_t smem = kWarps * (kFixed + stage);
  return launch_staged<kStagedThreads>(true, rta_big_kernel<SLOTS, MODE>, blocks_by_registers, kWarps * (kFixed + kMost), smem,
                       kSmemPerSm / (smem + kSmemPerBlockReserved), (p.n_tasksets + kWarps - 1) / kWarps, sm_count, st, p,
                       bin, (u32)stage);
}

template <bool LARGE, int MODE>
cudaError_t launch_deferred(const KParams &p, int sm_count, cudaStream_t st) {
  constexpr int kWarps = kBlockThreads / 32;
  static int blocks_per_sm[64] = {0};
  const size_t smem = sizeof(u32) * deferred_warp_words<LARGE>() * kWarps;
  return launch_persistent_ex(true, rta_deferred_kernel<LARGE, MODE>, blocks_per_sm, smem,
                              (p.n_tasksets + kWarps - 1) / kWarps, sm_count, st, p);
}

cudaError_t launch_plan_behind_tiles(const KParams &p, int sm_count, cudaStream_t st) {
  const i64 blocks = (p.n_tasksets + kPlanItems - 1) / kPlanItems, most = (i64)sm_count * 8;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned int)(blocks < most ? blocks : most)), cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr, cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, plan_behind_tiles_kernel, p);
}

template <int MODE>
cudaError_t launch_all_bins(const KParams &p, int sm_count, cudaStream_t st) {
  constexpr int kWarps = kBlockThreads / 32;
  static int blocks_per_sm[64] = {0};
  const size_t smem = sizeof(u32) * kSmallWarpWords * kWarps;
  cudaError_t e = launch_persistent(rta_small_kernel<MODE>, blocks_per_sm, smem,
                                    (p.n_tasksets + kWarps - 1) / kWarps, sm_count, st, p);
  if (e == cudaSuccess) e = launch_big<2, MODE>(p, 4, sm_count, st);
  if (e == cudaSuccess) e = launch_big<3, MODE>(p, 5, sm_count, st);
  if (e == cudaSuccess) e = launch_big<4, MODE>(p, 6, sm_count, st);
  if (e == cudaSuccess) e = launch_big<6, MODE>(p, 7, sm_count, st);
  if (e == cudaSuccess) e = launch_big<8, MODE>(p, 8, sm_count, st);
  if (e == cudaSuccess) e = launch_deferred<false, MODE>(p, sm_count, st);
  if (e == cudaSuccess) e = launch_deferred<true, MODE>(p, sm_count, st);
  return e;
}

// Tiles are for batches of tasksets of one size, whose mean is a whole number; where that is a mixture's all the same, the tile
// kernel finds out (tile_batch).  Under GCAPS a tile's walk is long, so there have to be enough tiles to go round: 12 tasks 43 / 54 us (tiles /
// bins) at 12,500 tasksets and 63 / 84 at 50,000, 16 tasks 71 / 69 at 25,000 and 79 / 83 at 35,000, 20 tasks 91 / 84
// and 97 / 105, 24 tasks 127 / 123 at 35,000 and 128 / 157 at 50,000.  Under RR tiles are the faster way from the start
// (24 tasks 40 / 51 us at 12,500).  Several analyses under GCAPS, 20 tasks: 170 / 138 us for five pairs of 10,000
// tasksets, 243 / 240 of 20,000, 212 / 280 for three pairs of 50,000; 24 tasks: 203 / 182 for two pairs of 30,000, 578 / 654 for
// 25 pairs of 5,000.  32 tasks: 575 / 521 us per 100,000, as a tile then takes 40 KB.
// Returns how many tasks the tasksets have, or 0: no tiles.  `analyses`: those of the call; `walks`: how many of a policy
// every taskset goes through.
int tile_tasks(int analyses, int walks, i64 max_ovh, const KParams &p) {
  if (max_ovh >= (1 << 20) || ((analyses & 2) && (p.policy & GCAPS_RTA_LITERAL))) return 0;
  if (p.n_tasks % p.n_tasksets != 0 || p.n_tasks > kTileMost * p.n_tasksets) return 0;
  const int n = (int)(p.n_tasks / p.n_tasksets);
  if (walks == 1 && (analyses & 3) && n > 12 && p.n_tasksets < 1750 * n) return 0;
  if (walks > 1 && (analyses & 12) == 0 && n > 12 && p.n_tasksets * walks < 100000) return 0;
  return n;
}

// Whether the analyses of GCAPS and of RR go through tiles one after the other.  A kernel of both stages a tile once for all, but the more its
// walks have to do the more it loses to instruction fetch (it holds the walks twice) and to its shared memory.  Together / apart (by bins
// for the groups of lanes), 100,000 tasksets at U/core 0.5, 60 % GPU tasks: all four analyses of 16 tasks 330 / 355 us, 20 tasks 493 / 475,
// 22 tasks 589 / 537 (611), 24 tasks 842 / 656 (652); three pairs of two analyses, four lanes per taskset, of 12 tasks 330 / 344,
// 16 tasks 513 / 462 (553), 20 tasks 810 / 666 (755), 24 tasks 1,366 / 931 (862).  Small batches stay together, as GCAPS alone does
// not take tiles there (20 tasks, 15,000 tasksets, three pairs of four analyses: 350 / 365; 24 tasks, 30,000, of two: 369 / 330).
bool tiles_apart(int n, int walks, i64 n_tasksets) {
  return n > (walks > kKeptFew ? 12 : 22) && n_tasksets * walks >= (n > 22 ? 80000 : 100000);
}

// Plan + analysis launches of one call.  `sw` null: one analysis (p.policy).  Otherwise the
// analyses named in `analyses` (bit m = mode m) for every pair of `sw`: the self-suspension
// modes in one set of launches, the busy-waiting modes in another (the plan is shared, the work
// counters are cleared in between).
int enqueue_batch(KParams p, void *workspace, size_t workspace_bytes, int sm_count, cudaStream_t st,
                  const SweepArgs *sw = nullptr, int analyses = 0) {
  if (p.n_tasksets == 0) return GCAPS_OK;
  if (sw && sw->n == 1 && (analyses & (analyses - 1)) == 0 && p.out_wcrt && p.n_tasksets > kDirectSweepMost) {
    // one analysis once is what the kernels of a single analysis do
    p.policy = (p.policy & ~(0xff | GCAPS_RTA_BUSY)) | (analyses >= 4 ? GCAPS_POLICY_RR : GCAPS_POLICY_GCAPS) |
               ((analyses & 10) ? GCAPS_RTA_BUSY : 0);
    sw = nullptr;
  }
  const bool rr = (p.policy & 0xff) == GCAPS_POLICY_RR, busy = (p.policy & GCAPS_RTA_BUSY) != 0;
  const int mode = (rr ? 2 : 0) + (busy ? 1 : 0);
  const bool direct = p.n_tasksets <= (sw ? kDirectSweepMost : kDirectMost);
  const int rc = place_plan(p, workspace, workspace_bytes);
  if (rc != GCAPS_OK) return rc;
  // walks of a taskset through the recurrence that a tile's lanes share.  (A single one of GCAPS and of RR each is better
  // left to the groups of lanes, which stage once for both: 288 us for 100,001 tasksets of 20 tasks, 323 in tiles.)
  auto walks_of = [&](int which) -> int { return sw ? sw->n * (((which & 3) == 3 || (which & 12) == 12) ? 2 : 1) : 1; };
  auto tiles_of = [&](int which, int walks) -> int {
    return direct || (sw && walks == 1) ? 0 : tile_tasks(which, walks, sw ? sw->max_ovh : p.ovh, p);
  };
  const int all = sw ? analyses : 1 << mode;
  const int tile_n = tiles_of(all, walks_of(all));
  cudaError_t e = cudaGetLastError();
  // the plan, or the header that tiles start from
  auto begin = [&](int n) -> cudaError_t {
    if (n > 0) return cudaMemsetAsync(p.hdr, 0, sizeof(PlanHeader), st);
    if (!direct) enqueue_plan_kernels(p, st);
    return cudaGetLastError();
  };
  if (e == cudaSuccess && sw) {
    SweepArgs set = *sw;
    set.block_stride = __builtin_popcount(analyses);
    for (int m = 0, k = 0; m < 4; ++m) {
      set.block_of_mode[m] = k;
      k += (analyses >> m) & 1;
    }
    auto analyse = [&](int which, int walks, int n) -> cudaError_t {
      cudaError_t err = begin(n);
      if (n > 0) {
        set.enabled = which;
        if (err == cudaSuccess) err = walks > kKeptFew ? launch_tile_q4(p, set, n, sm_count, st) : launch_tile_q2(p, set, n, sm_count, st);
        if (err == cudaSuccess) err = launch_plan_behind_tiles(p, sm_count, st);
      }
      bool first = true;
      for (int half = 0; half < 2 && err == cudaSuccess; ++half) {
        set.enabled = which & (half == 0 ? 5 : 10);
        if (set.enabled == 0) continue;
        if (!first && !direct) err = cudaMemsetAsync(p.hdr->next, 0, sizeof(p.hdr->next), st);
        first = false;
        if (err == cudaSuccess)
          err = direct  ? launch_sweep_one_warp_each(p, set, sm_count, st)
                : n > 0 ? launch_sweep_rest(p, set, sm_count, st)
                        : launch_sweep_set(p, set, sm_count, st);
      }
      return err;
    };
    const int gcaps = analyses & 3, rr_ones = analyses & 12, gcaps_walks = walks_of(gcaps), rr_walks = walks_of(rr_ones);
    if (tile_n > 0 && gcaps && rr_ones && gcaps_walks > 1 && rr_walks > 1 && tiles_apart(tile_n, walks_of(all), p.n_tasksets)) {
      e = analyse(gcaps, gcaps_walks, tiles_of(gcaps, gcaps_walks));
      if (e == cudaSuccess) e = analyse(rr_ones, rr_walks, tiles_of(rr_ones, rr_walks));
    } else {
      e = analyse(analyses, walks_of(all), tile_n);
    }
  } else if (e == cudaSuccess && tile_n > 0) {
    e = begin(tile_n);
    if (e == cudaSuccess) e = launch_tiles(mode, p, tile_n, sm_count, st);
    if (e == cudaSuccess) e = launch_plan_behind_tiles(p, sm_count, st);
    if (e == cudaSuccess) e = launch_rest(mode, p, sm_count, st);
  } else if (e == cudaSuccess) {
    e = begin(0);
    if (e == cudaSuccess)
      e = direct      ? launch_one_warp_each(mode, p, st)
          : mode == 0 ? launch_all_bins<0>(p, sm_count, st)
          : mode == 1 ? launch_all_bins<1>(p, sm_count, st)
          : mode == 2 ? launch_all_bins<2>(p, sm_count, st)
                      : launch_all_bins<3>(p, sm_count, st);
  }
  if (e != cudaSuccess) {
    g_last_cuda_error = (int)e;
    return GCAPS_ERR_CUDA;
  }
  return GCAPS_OK;
}

// staging memory of the host-buffer entry point (one set per process, current device)
constexpr int kStageSlots = 3;  // one chunk on its way in, one analysed, one on its way out
struct HostStage {
  void *dev[kStageSlots];
  size_t dev_bytes[kStageSlots];
  cudaStream_t stream[kStageSlots];
  int device;
  bool streams_ok;
};
HostStage g_stage = {{nullptr}, {0}, {nullptr}, -1, false};
std::mutex g_stage_mutex;  // one host-buffer call at a time owns the staging slots

void release_stage_locked() {
  for (int k = 0; k < kStageSlots; ++k) {
    if (g_stage.dev[k]) cudaFree(g_stage.dev[k]);
    g_stage.dev[k] = nullptr;
    g_stage.dev_bytes[k] = 0;
    if (g_stage.streams_ok && g_stage.stream[k]) cudaStreamDestroy(g_stage.stream[k]);
    g_stage.stream[k] = nullptr;
  }
  g_stage.streams_ok = false;
  g_stage.device = -1;
}

// Workspace of gcaps_rta_batch_static: lives in the library image, one copy per device that
// loads it.  In host code this name is only a handle for cudaGetSymbolAddress, never an address
// a kernel may be given.
static __device__ __align__(256) unsigned char g_static_scratch[GCAPS_RTA_STATIC_SCRATCH_BYTES];
void *g_static_scratch_ptr[64];  // device address of the array, per device, once looked up

}  // namespace

extern "C" {

size_t gcaps_rta_workspace_bytes(int64_t n_tasksets) {
  if (n_tasksets <= 0) return 0;
  const size_t nb = plan_blocks(n_tasksets);
  return 256 + align_up(nb * kBinStride * sizeof(unsigned int), 256) +
         align_up((size_t)n_tasksets * sizeof(unsigned int), 256);
}

int gcaps_rta_batch(const gcaps_tasksets_t *ts, int64_t n_tasksets, int policy,
                    int64_t timeslice_us, int64_t ctx_switch_overhead_us, int64_t *out_wcrt,
                    uint8_t *out_sched, void *workspace, size_t workspace_bytes, void *stream) {
  int rc = check_args(ts, n_tasksets, policy, timeslice_us, ctx_switch_overhead_us);
  if (rc != GCAPS_OK) return rc;
  if (n_tasksets == 0) return GCAPS_OK;
  if (!out_sched || (ts->n_tasks > 0 && !out_wcrt)) return GCAPS_ERR_INVALID_ARG;
  DeviceInfo di;
  rc = device_info(&di);
  if (rc != GCAPS_OK) return rc;
  KParams p;
  fill_params(&p, ts, n_tasksets, policy, timeslice_us, ctx_switch_overhead_us, out_wcrt, out_sched);
  return enqueue_batch(p, workspace, workspace_bytes, di.sm_count, (cudaStream_t)stream);
}

int gcaps_rta_multi_batch(const gcaps_tasksets_t *ts, int64_t n_tasksets, int analyses, int flags,
                          int n_points, const int64_t *timeslice_us,
                          const int64_t *ctx_switch_overhead_us, int64_t *out_wcrt,
                          uint8_t *out_sched, void *workspace, size_t workspace_bytes, void *stream) {
  if (analyses < 1 || analyses > 15 || (flags & ~(GCAPS_RTA_LITERAL | GCAPS_RTA_BEST_EFFORT)))
    return GCAPS_ERR_INVALID_ARG;
  if (n_points < 1 || n_points > GCAPS_RTA_MAX_SWEEP || !ctx_switch_overhead_us)
    return GCAPS_ERR_INVALID_ARG;
  const bool rr = (analyses & (GCAPS_ANALYSIS_RR_SUSPEND | GCAPS_ANALYSIS_RR_BUSY)) != 0;
  if (rr && !timeslice_us) return GCAPS_ERR_INVALID_ARG;
  const int policy = (rr ? GCAPS_POLICY_RR : GCAPS_POLICY_GCAPS) | flags;  // (for the argument checks)
  SweepArgs sw;
  memset(&sw, 0, sizeof(sw));
  sw.n = n_points;
  for (int q = 0; q < n_points; ++q) {
    const int64_t L = rr ? timeslice_us[q] : 1;
    int rc = check_args(ts, n_tasksets, policy, L, ctx_switch_overhead_us[q]);
    if (rc != GCAPS_OK) return rc;
    KParams one;  // (fills the reciprocal of L exactly as a single call would)
    fill_params(&one, ts, n_tasksets, policy, L, ctx_switch_overhead_us[q], nullptr, nullptr);
    sw.q[q].L = one.L, sw.q[q].ovh = one.ovh;
    sw.q[q].l_mode = one.l_mode, sw.q[q].l_magic = one.l_magic, sw.q[q].l_shift = one.l_shift;
    if (one.ovh > sw.max_ovh) sw.max_ovh = one.ovh;
  }
  if (n_tasksets == 0) return GCAPS_OK;
  if (!out_sched) return GCAPS_ERR_INVALID_ARG;
  DeviceInfo di;
  int rc = device_info(&di);
  if (rc != GCAPS_OK) return rc;
  KParams p;
  fill_params(&p, ts, n_tasksets, policy, sw.q[0].L, sw.q[0].ovh, out_wcrt, out_sched);
  return enqueue_batch(p, workspace, workspace_bytes, di.sm_count, (cudaStream_t)stream, &sw, analyses);
}

int gcaps_rta_sweep_batch(const gcaps_tasksets_t *ts, int64_t n_tasksets, int policy, int n_points,
                          const int64_t *timeslice_us, const int64_t *ctx_switch_overhead_us,
                          int64_t *out_wcrt, uint8_t *out_sched, void *workspace,
                          size_t workspace_bytes, void *stream) {
  const int pol = policy & 0xff;
  if (pol != GCAPS_POLICY_GCAPS && pol != GCAPS_POLICY_RR) return GCAPS_ERR_INVALID_ARG;
  if (policy & ~(0xff | GCAPS_RTA_BUSY | GCAPS_RTA_LITERAL | GCAPS_RTA_BEST_EFFORT)) return GCAPS_ERR_INVALID_ARG;
  const int mode = (pol == GCAPS_POLICY_RR ? 2 : 0) + ((policy & GCAPS_RTA_BUSY) ? 1 : 0);
  return gcaps_rta_multi_batch(ts, n_tasksets, 1 << mode, policy & (GCAPS_RTA_LITERAL | GCAPS_RTA_BEST_EFFORT),
                               n_points, timeslice_us, ctx_switch_overhead_us, out_wcrt, out_sched,
                               workspace, workspace_bytes, stream);
}

int gcaps_rta_batch_static(const gcaps_tasksets_t *ts, int64_t n_tasksets, int policy,
                           int64_t timeslice_us, int64_t ctx_switch_overhead_us,
                           int64_t *out_wcrt, uint8_t *out_sched, void *stream) {
  int rc = check_args(ts, n_tasksets, policy, timeslice_us, ctx_switch_overhead_us);
  if (rc != GCAPS_OK) return rc;
  if (n_tasksets > GCAPS_RTA_STATIC_MAX_TASKSETS ||
      gcaps_rta_workspace_bytes(n_tasksets) > (size_t)GCAPS_RTA_STATIC_SCRATCH_BYTES)
    return GCAPS_ERR_TOO_LARGE;
  if (n_tasksets == 0) return GCAPS_OK;
  if (!out_sched || (ts->n_tasks > 0 && !out_wcrt)) return GCAPS_ERR_INVALID_ARG;
  DeviceInfo di;
  rc = device_info(&di);
  if (rc != GCAPS_OK) return rc;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 64) {
    g_last_cuda_error = (int)e;
    return GCAPS_ERR_NO_DEVICE;
  }
  void *scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_init_mutex);
    if (!g_static_scratch_ptr[dev]) {
      // once per device, with that device current: the array's address on this device
      void *ptr = nullptr;
      e = cudaGetSymbolAddress(&ptr, g_static_scratch);
      if (e != cudaSuccess || !ptr) {
        g_last_cuda_error = (int)e;
        return GCAPS_ERR_CUDA;
      }
      g_static_scratch_ptr[dev] = ptr;
    }
    scratch = g_static_scratch_ptr[dev];
  }
  KParams p;
  fill_params(&p, ts, n_tasksets, policy, timeslice_us, ctx_switch_overhead_us, out_wcrt, out_sched);
  // Nothing in the array has to be cleared first: the header (counts, starts, work counters) is written by the plan kernels or,
  // in front of tiles, cleared in the stream, and every per-block count and permutation entry that a kernel of
  // this call reads is written by one before it.
  return enqueue_batch(p, scratch, (size_t)GCAPS_RTA_STATIC_SCRATCH_BYTES, di.sm_count,
                       (cudaStream_t)stream);
}

int gcaps_rta_batch_few(const gcaps_tasksets_t *ts, int64_t n_tasksets, int policy, int64_t timeslice_us,
                        int64_t ctx_switch_overhead_us, int64_t *out_wcrt, uint8_t *out_sched, void *stream) {
  static_assert(GCAPS_RTA_FEW_MAX_TASKSETS == kDirectMost, "what runs as one launch");
  int rc = check_args(ts, n_tasksets, policy, timeslice_us, ctx_switch_overhead_us);
  if (rc != GCAPS_OK) return rc;
  if (n_tasksets > GCAPS_RTA_FEW_MAX_TASKSETS) return GCAPS_ERR_TOO_LARGE;
  if (n_tasksets == 0) return GCAPS_OK;
  if (!out_sched || (ts->n_tasks > 0 && !out_wcrt)) return GCAPS_ERR_INVALID_ARG;
  DeviceInfo di;
  rc = device_info(&di);
  if (rc != GCAPS_OK) return rc;
  KParams p;
  fill_params(&p, ts, n_tasksets, policy, timeslice_us, ctx_switch_overhead_us, out_wcrt, out_sched);
  const bool rr = (policy & 0xff) == GCAPS_POLICY_RR, busy = (policy & GCAPS_RTA_BUSY) != 0;
  const cudaError_t e = launch_one_warp_each((rr ? 2 : 0) + (busy ? 1 : 0), p, (cudaStream_t)stream);
  if (e != cudaSuccess) {
    g_last_cuda_error = (int)e;
    return GCAPS_ERR_CUDA;
  }
  return GCAPS_OK;
}

int gcaps_rta_validate(const gcaps_tasksets_t *ts, int64_t n_tasksets, int32_t *out_err,
                       void *stream) {
  int rc = check_args(ts, n_tasksets, GCAPS_POLICY_GCAPS, 1, 0);
  if (rc != GCAPS_OK) return rc;
  if (n_tasksets == 0) return GCAPS_OK;
  if (!out_err) return GCAPS_ERR_INVALID_ARG;
  DeviceInfo di;
  rc = device_info(&di);
  if (rc != GCAPS_OK) return rc;
  KParams p;
  fill_params(&p, ts, n_tasksets, GCAPS_POLICY_GCAPS, 1, 0, nullptr, nullptr);
  validate_kernel<<<(unsigned int)((n_tasksets + 127) / 128), 128, 0, (cudaStream_t)stream>>>(p, out_err);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    g_last_cuda_error = (int)e;
    return GCAPS_ERR_CUDA;
  }
  return GCAPS_OK;
}

#define HOST_TRY(call)                    \
  do {                                    \
    cudaError_t e_ = (call);              \
    if (e_ != cudaSuccess) {              \
      g_last_cuda_error = (int)e_;        \
      return GCAPS_ERR_CUDA;              \
    }                                     \
  } while (0)

void gcaps_rta_release_host(void) {
  std::lock_guard<std::mutex> lock(g_stage_mutex);
  release_stage_locked();
}

constexpr int kMaxHostPolicies = GCAPS_RTA_MAX_HOST_POLICIES;

// Copies tasksets [t, t1) (tasks [k0, k1)) to the staging slot, enqueues their analysis under
// every requested policy and the copies of the results back.  The offsets of the range are known to be monotone and in range.
static int host_chunk(const gcaps_tasksets_t *ts, int64_t t, int64_t t1, const int *policies,
                      int n_pol, int64_t L, int64_t ovh, int64_t *const *out_wcrt,
                      uint8_t *const *out_sched, int slot, int sm_count) {
  const int64_t k0 = ts->task_off[t], k1 = ts->task_off[t1];
  const int64_t nt = t1 - t, nk = k1 - k0;
  const int64_t c0 = ts->cseg_off[k0], nc = ts->cseg_off[k1] - c0;
  const int64_t g0 = ts->gseg_off[k0], ng = ts->gseg_off[k1] - g0;
  size_t off = 0;
  auto take = [&](size_t n_bytes) {
    size_t o = off;
    off += align_up(n_bytes, 256);
    return o;
  };
  const size_t o_task_off = take((nt + 1) * 8), o_period = take(nk * 8), o_deadline = take(nk * 8);
  const size_t o_priority = take(nk * 8), o_core = take(nk * 8), o_cseg_off = take((nk + 1) * 8);
  const size_t o_cseg = take(nc * 8), o_gseg_off = take((nk + 1) * 8), o_gm = take(ng * 8);
  const size_t o_ge = take(ng * 8);
  size_t o_wcrt[kMaxHostPolicies], o_sched[kMaxHostPolicies];
  for (int q = 0; q < n_pol; ++q) o_wcrt[q] = take(nk * 8), o_sched[q] = take(nt);
  const size_t ws_bytes = gcaps_rta_workspace_bytes(nt);
  const size_t o_ws = take(ws_bytes);
  cudaStream_t st = g_stage.stream[slot];
  HOST_TRY(cudaStreamSynchronize(st));  // the slot's previous chunk has left the buffer
  if (g_stage.dev_bytes[slot] < off) {
    if (g_stage.dev[slot]) HOST_TRY(cudaFree(g_stage.dev[slot]));
    g_stage.dev[slot] = nullptr;
    g_stage.dev_bytes[slot] = 0;
    const size_t want = off + (off >> 3);
    HOST_TRY(cudaMalloc(&g_stage.dev[slot], want));
    g_stage.dev_bytes[slot] = want;
  }
  unsigned char *d = (unsigned char *)g_stage.dev[slot];
#define H2D(dst_off, src, count) \
  HOST_TRY(cudaMemcpyAsync(d + (dst_off), (src), (size_t)(count) * 8, cudaMemcpyHostToDevice, st))
  H2D(o_task_off, ts->task_off + t, nt + 1);
  if (nk > 0) {
    H2D(o_period, ts->period + k0, nk);
    H2D(o_deadline, ts->deadline + k0, nk);
    H2D(o_priority, ts->priority + k0, nk);
    H2D(o_core, ts->core + k0, nk);
  }
  H2D(o_cseg_off, ts->cseg_off + k0, nk + 1);
  H2D(o_gseg_off, ts->gseg_off + k0, nk + 1);
  if (nc > 0) H2D(o_cseg, ts->cseg_wcet + c0, nc);
  if (ng > 0) {
    H2D(o_gm, ts->gseg_misc + g0, ng);
    H2D(o_ge, ts->gseg_exec + g0, ng);
  }
#undef H2D
  gcaps_tasksets_t dts;
  dts.n_tasks = nk, dts.n_csegs = nc, dts.n_gsegs = ng;
  dts.task_off = (const int64_t *)(d + o_task_off);
  dts.period = (const int64_t *)(d + o_period);
  dts.deadline = (const int64_t *)(d + o_deadline);
  dts.priority = (const int64_t *)(d + o_priority);
  dts.core = (const int64_t *)(d + o_core);
  dts.cseg_off = (const int64_t *)(d + o_cseg_off);
  dts.cseg_wcet = (const int64_t *)(d + o_cseg);
  dts.gseg_off = (const int64_t *)(d + o_gseg_off);
  dts.gseg_misc = (const int64_t *)(d + o_gm);
  dts.gseg_exec = (const int64_t *)(d + o_ge);
  for (int q = 0; q < n_pol; ++q) {  // one copy of the inputs, one analysis per policy
    KParams p;
    fill_params(&p, &dts, nt, policies[q], L, ovh, (int64_t *)(d + o_wcrt[q]), d + o_sched[q]);
    p.task_base = k0, p.cseg_base = c0, p.gseg_base = g0;
    int rc = enqueue_batch(p, d + o_ws, ws_bytes, sm_count, st);
    if (rc != GCAPS_OK) return rc;
    if (nk > 0)
      HOST_TRY(cudaMemcpyAsync(out_wcrt[q] + k0, d + o_wcrt[q], (size_t)nk * 8,
                               cudaMemcpyDeviceToHost, st));
    HOST_TRY(cudaMemcpyAsync(out_sched[q] + t, d + o_sched[q], (size_t)nt, cudaMemcpyDeviceToHost, st));
  }
  return GCAPS_OK;
}

// An error in a later chunk: earlier chunks' copies into the caller's arrays may still be in
// flight on the staging streams; nothing of this call may touch the caller's memory once it has
// returned.  Keeps the CUDA error code the failing step recorded.
static int drain_stage(int rc) {
  const int keep = g_last_cuda_error;
  for (int k = 0; k < kStageSlots; ++k)
    if (g_stage.streams_ok && g_stage.stream[k]) cudaStreamSynchronize(g_stage.stream[k]);
  g_last_cuda_error = keep;
  return rc;
}

// True if the task range [k0, k1] is inside the arrays and both segment offset arrays are
// non-decreasing and in range over it.
static bool host_range_is_canonical(const gcaps_tasksets_t *ts, int64_t k0, int64_t k1) {
  if (k0 < 0 || k1 < k0 || k1 > ts->n_tasks) return false;
  if (ts->cseg_off[k0] < 0 || ts->cseg_off[k1] > ts->n_csegs) return false;
  if (ts->gseg_off[k0] < 0 || ts->gseg_off[k1] > ts->n_gsegs) return false;
  // a negative value or step sets the sign bit (no step between non-negative values overflows)
  int64_t sign = 0;
  for (int64_t k = k0; k < k1; ++k)
    sign |= ts->cseg_off[k + 1] | ts->gseg_off[k + 1] | (int64_t)((uint64_t)ts->cseg_off[k + 1] - (uint64_t)ts->cseg_off[k]) |
            (int64_t)((uint64_t)ts->gseg_off[k + 1] - (uint64_t)ts->gseg_off[k]);
  return sign >= 0;
}

int gcaps_rta_batch_host(const gcaps_tasksets_t *ts, int64_t n_tasksets, int policy,
                         int64_t timeslice_us, int64_t ctx_switch_overhead_us, int64_t *out_wcrt,
                         uint8_t *out_sched) {
  return gcaps_rta_batch_host_multi(ts, n_tasksets, &policy, 1, timeslice_us, ctx_switch_overhead_us,
                                    &out_wcrt, &out_sched);
}

int gcaps_rta_batch_host_multi(const gcaps_tasksets_t *ts, int64_t n_tasksets, const int *policies,
                               int n_policies, int64_t timeslice_us, int64_t ctx_switch_overhead_us,
                               int64_t *const *out_wcrt, uint8_t *const *out_sched) {
  if (!policies || n_policies < 1 || n_policies > kMaxHostPolicies || !out_wcrt || !out_sched)
    return GCAPS_ERR_INVALID_ARG;
  int rc = GCAPS_OK;
  for (int q = 0; q < n_policies; ++q) {
    rc = check_args(ts, n_tasksets, policies[q], timeslice_us, ctx_switch_overhead_us);
    if (rc != GCAPS_OK) return rc;
  }
  if (n_tasksets == 0) return GCAPS_OK;
  for (int q = 0; q < n_policies; ++q)
    if (!out_sched[q] || (ts->n_tasks > 0 && !out_wcrt[q])) return GCAPS_ERR_INVALID_ARG;
  DeviceInfo di;
  rc = device_info(&di);
  if (rc != GCAPS_OK) return rc;
  std::lock_guard<std::mutex> lock(g_stage_mutex);
  int dev = 0;
  HOST_TRY(cudaGetDevice(&dev));
  if (g_stage.device != dev) {
    release_stage_locked();
    g_stage.device = dev;
  }
  if (!g_stage.streams_ok) {
    for (int k = 0; k < kStageSlots; ++k)
      HOST_TRY(cudaStreamCreateWithFlags(&g_stage.stream[k], cudaStreamNonBlocking));
    g_stage.streams_ok = true;
  }
  const int64_t kChunkTasksets = 1 << 16;
  // What the first chunk's checks, the last chunk's analysis and its way back take is not hidden behind a
  // transfer, so the chunks of a short batch are small (256 k tasks, 30 MB, 0.6 ms of the host link:
  // 60,000 80-task tasksets, two policies, page-locked arrays: 15.4 -> 12.0 ms against chunks of up to
  // 3 M tasks); every chunk costs its ten copies and its launches, so those of a long one are larger
  // (300,000 such tasksets: 54.8 ms; 58.5 in chunks of 256 k, 56.1 in chunks of 3 M tasks).
  int64_t chunk_tasks = ts->n_tasks / 24;
  chunk_tasks = chunk_tasks < (1 << 18) ? (1 << 18) : chunk_tasks > (1 << 21) ? (1 << 21) : chunk_tasks;
  int64_t t = 0;
  int slot = 0;
  while (t < n_tasksets) {
    // a chunk is a run of whole tasksets whose task ranges follow one another
    int64_t t1 = t;
    const int64_t k0 = ts->task_off[t];
    int64_t k1 = k0;
    while (t1 < n_tasksets && t1 - t < kChunkTasksets) {
      const int64_t kn = ts->task_off[t1 + 1];
      if (kn < k1 || (t1 > t && kn - k0 > chunk_tasks)) break;
      k1 = kn;
      t1 += 1;
    }
    if (t1 > t && host_range_is_canonical(ts, k0, k1)) {
      rc = host_chunk(ts, t, t1, policies, n_policies, timeslice_us, ctx_switch_overhead_us,
                      out_wcrt, out_sched, slot, di.sm_count);
      if (rc != GCAPS_OK) return drain_stage(rc);
      slot = (slot + 1) % kStageSlots;
      t = t1;
      continue;
    }
    // Malformed offsets somewhere in the run: go through it one taskset at a time, so that each
    // taskset is judged on its own offsets alone.
    const int64_t stop = t1 > t ? t1 : t + 1;
    for (; t < stop; ++t) {
      const int64_t a = ts->task_off[t], b = ts->task_off[t + 1];
      if (a < 0 || b < a || b > ts->n_tasks || b - a > GCAPS_RTA_MAX_TASKS) {
        for (int q = 0; q < n_policies; ++q) out_sched[q][t] = GCAPS_SCHED_INVALID;
      } else if (!host_range_is_canonical(ts, a, b)) {
        for (int q = 0; q < n_policies; ++q) {
          out_sched[q][t] = GCAPS_SCHED_INVALID;
          for (int64_t k = a; k < b; ++k) out_wcrt[q][k] = GCAPS_WCRT_INVALID;
        }
      } else {
        rc = host_chunk(ts, t, t + 1, policies, n_policies, timeslice_us, ctx_switch_overhead_us,
                        out_wcrt, out_sched, slot, di.sm_count);
        if (rc != GCAPS_OK) return drain_stage(rc);
        slot = (slot + 1) % kStageSlots;
      }
    }
  }
  for (int k = 0; k < kStageSlots; ++k) HOST_TRY(cudaStreamSynchronize(g_stage.stream[k]));
  return GCAPS_OK;
}

const char *gcaps_rta_strerror(int code) {
  switch (code) {
    case GCAPS_OK: return "ok";
    case GCAPS_ERR_INVALID_ARG: return "invalid argument";
    case GCAPS_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
    case GCAPS_ERR_CUDA: return "CUDA runtime error (see gcaps_rta_last_cuda_error)";
    case GCAPS_ERR_NO_DEVICE: return "no usable sm_100 CUDA device";
    case GCAPS_ERR_TOO_LARGE:
      return "batch exceeds the limit of this entry point (GCAPS_RTA_STATIC_MAX_TASKSETS, GCAPS_RTA_FEW_MAX_TASKSETS): split it or use gcaps_rta_batch";
    default: return "unknown error code";
  }
}

int gcaps_rta_last_cuda_error(void) { return g_last_cuda_error; }

int gcaps_rta_version(void) { return GCAPS_RTA_VERSION; }

}  // extern "C"
