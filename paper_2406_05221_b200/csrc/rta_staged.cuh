// rta_staged.cuh -- one analysis per taskset, staged into shared memory by asynchronous bulk copies.
// Internal; included by gcaps_rta.cu.
//
// A warp owns a stage: room for the nine slices (six per-task arrays, three segment arrays) of one
// taskset.  It looks at the first ranks of the priority order straight out of the staged data
// (staged_head), and as soon as what it needs from there is in registers and in the few rows of
// those ranks, the copies of its next taskset are on their way, before the recurrence runs and the
// results are written.  No load instruction waits for DRAM, no value passes through registers on its
// way into shared memory, and per-task sums are formed for the first ranks only: where tasksets are
// far from schedulable (the first deadline miss comes within 16 ranks for all but 0.02 % of the `large`
// and `divergence` tasksets) that is all there is to do.  Every value of the taskset is still read and
// range-checked.  A taskset that none of these ranks decides, or that this kernel cannot take (too
// many segments for a stage, values beyond the 32-bit path, at the very end of an array), takes the full
// pass: at the end of the warp's own work while there are few, else it is marked in the permutation and
// left to a second launch (run_deferred_bin), which needs no stages and so has more warps for the
// recurrence.  Which of the two is staged_walk.h.
//
// 1,000,000 `large` tasksets (9.75 GB in and out): GCAPS 2.39 -> 1.58 ms, round robin 2.18 -> 1.52 ms
// (6.2 and 6.4 TB/s): bound by HBM.  Before, 1,775 warp instructions per taskset and the latency of
// its own loads kept a warp busy; the same look at the first ranks with plain loads had gained
// nothing under GCAPS (with less arithmetic between a taskset's loads, 24 warps did not cover their
// latency).
#ifndef GCAPS_RTA_STAGED_CUH_
#define GCAPS_RTA_STAGED_CUH_

#include <cuda_runtime.h>
#include <stdint.h>

#include "rta_device.cuh"
#include "staged_walk.h"

namespace {

constexpr int kStagedThreads = kStagedBlockThreads;  // two warps: the number of stages per SM adapts finely
constexpr int kHeadRanks = 16;  // two lanes per rank
constexpr int kStagedChunk = 8;  // tasksets of one pull
constexpr int kArrays = 9;       // period, deadline, priority, core, cseg_off, gseg_off, cseg, gm, ge
constexpr int kHeadUndecided = 2;
constexpr u32 kStageWaitLimit = 1u << 20;  // polls (each up to a hardware time slice) before giving up

// rows of the first ranks, in the form recurrence_narrow reads
struct HeadRows {
  unsigned char *buf;
  __device__ __forceinline__ uint4 &a(int r) const { return reinterpret_cast<uint4 *>(buf)[r]; }
  __device__ __forceinline__ uint4 &b(int r) const { return reinterpret_cast<uint4 *>(buf)[kHeadRanks + r]; }
  __device__ __forceinline__ u32 &base(int r) const { return reinterpret_cast<u32 *>(buf + 32 * kHeadRanks)[r]; }
  __device__ __forceinline__ u32 &R(int r) const { return reinterpret_cast<u32 *>(buf + 36 * kHeadRanks)[r]; }
};

// Shared memory of one warp, in front of its stage.
template <int SLOTS>
struct __align__(16) StagedWarp {
  Ahead ahead[2 * kStagedChunk];
  __align__(16) unsigned char rows[40 * kHeadRanks];
  u32 left[kLeftMost];  // entries of the bin
  __align__(16) u32 offset[12];  // where in the stage each array's slice starts; [9]: where all end
  __align__(16) unsigned char pos_of_rank[32 * SLOTS];
  __align__(16) unsigned long long barrier;
};

// blocks per SM the register allocation aims at
__host__ __device__ constexpr int staged_min_blocks(int slots) { return slots <= 3 ? 10 : slots == 4 ? 8 : 5; }

struct SliceTable {
  const i64 *ptr[kArrays];
  i64 len[kArrays];
};

__device__ __forceinline__ u32 smem_addr(const void *ptr) { return (u32)__cvta_generic_to_shared(ptr); }

__device__ __forceinline__ void barrier_init(unsigned long long *bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void barrier_expect(unsigned long long *bar, u32 bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
// Waits for the phase of the given parity; false if it has not completed after kStageWaitLimit polls.
__device__ __forceinline__ bool barrier_wait(unsigned long long *bar, u32 parity) {
  for (u32 k = 0; k < kStageWaitLimit; ++k) {
    u32 done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}
__device__ __forceinline__ void bulk_load(u32 dst, const void *src, u32 bytes, unsigned long long *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}

// Starts the copies of the taskset `me` into the warp's stage, one lane per array.  A copy must start
// and end on 16-byte boundaries, so a slice may bring one element of a neighbour along at either
// end.  False, with nothing started, if the slices do not fit the stage or such an end lies outside
// its array.
template <int SLOTS>
__device__ __forceinline__ bool stage_taskset(const SliceTable &tab, const Ahead &me, StagedWarp<SLOTS> &w,
                                              unsigned char *stage, u32 stage_bytes, int lane) {
  const int k = lane < kArrays ? lane : 0;
  const i64 n = (i64)(me.packed & 0x1ffu), nc = (i64)((me.packed >> 9) & 0x7ffu), ng = (i64)((me.packed >> 20) & 0x7ffu);
  const i64 first = k < 6 ? me.a : (k == 6 ? me.c_lo : me.g_lo);
  const i64 count = k < 4 ? n : (k < 6 ? n + 1 : (k == 6 ? nc : ng));
  const unsigned char *const array = reinterpret_cast<const unsigned char *>(tab.ptr[k]);
  const unsigned char *const slice = array + 8 * first;
  const u32 odd = (u32)((uintptr_t)slice & 8u);  // (int64 arrays: 8-byte aligned)
  const unsigned char *const src = slice - odd;
  const u32 bytes = (lane < kArrays && count > 0) ? ((odd + 8u * (u32)count + 15u) & ~15u) : 0u;
  const bool inside = bytes == 0 || (src >= array && src + bytes <= array + 8 * tab.len[k]);
  u32 end = bytes;
#pragma unroll
  for (int d = 1; d < 16; d <<= 1) {
    const u32 y = __shfl_up_sync(kFull, end, d);
    if (lane >= d) end += y;
  }
  const u32 total = __shfl_sync(kFull, end, kArrays - 1);
  if (!__all_sync(kFull, inside) || total > stage_bytes) return false;
  const u32 at = end - bytes;
  if (lane < kArrays) w.offset[lane] = at + odd;
  if (lane == kArrays) w.offset[kArrays] = total;
  // what the warp has read from and written to the stage comes before what the copies write
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  if (lane == 0) barrier_expect(&w.barrier, total);
  __syncwarp();
  if (bytes > 0) bulk_load(smem_addr(stage) + at, src, bytes, &w.barrier);
  return true;
}

// The first ranks of a staged taskset.  Returns kFastDone (outputs written) or kHeadUndecided (all of
// them converged, or something needs the full or the exact path).  `next`: called once, as soon as
// the stage may be overwritten.
template <int SLOTS, int MODE, class Next>
__device__ __forceinline__ int staged_head(const KParams &p, const Ahead &me, StagedWarp<SLOTS> &w,
                                           const unsigned char *stage, int lane, Next next) {
  constexpr bool kGcaps = MODE < 2;
  const bool literal = (p.policy & GCAPS_RTA_LITERAL) != 0;
  const bool best_effort = (p.policy & GCAPS_RTA_BEST_EFFORT) != 0;
  const int n = (int)(me.packed & 0x1ffu);
  const u32 ng = (me.packed >> 20) & 0x7ffu;
  const HeadRows rows{w.rows};
  const uint4 off0 = *reinterpret_cast<const uint4 *>(&w.offset[0]);
  const uint4 off1 = *reinterpret_cast<const uint4 *>(&w.offset[4]);
  const uint2 off2 = *reinterpret_cast<const uint2 *>(&w.offset[8]);
  const i64 *const sT = reinterpret_cast<const i64 *>(stage + off0.x);
  const i64 *const sD = reinterpret_cast<const i64 *>(stage + off0.y);
  const i64 *const sP = reinterpret_cast<const i64 *>(stage + off0.z);
  const i64 *const sK = reinterpret_cast<const i64 *>(stage + off0.w);
  const i64 *const sCo = reinterpret_cast<const i64 *>(stage + off1.x);
  const i64 *const sGo = reinterpret_cast<const i64 *>(stage + off1.y);

  // ---- range check of the per-task values ------------------------------------------------------
  // `bad`: some bit is set if a value does not fit the 32-bit path
  u32 bad = 0;
  bool ok = true;
  int prio[SLOTS], rank[SLOTS];
  bool uses_gpu[SLOTS];
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    const int i = lane + 32 * s < n ? lane + 32 * s : n - 1;  // (lanes behind the end repeat the last task)
    const i64 T = sT[i], D = sD[i], P = sP[i], K = sK[i];
    const i64 dc = sCo[i + 1] - sCo[i], dg = sGo[i + 1] - sGo[i];
    bad |= (u32)((u64)T >> 32) | (u32)((u64)D >> 32) | (u32)((u64)K >> 32);
    bad |= (u32)((u64)dc >> 32) | (u32)((u64)dg >> 32) | (((u32)dc | (u32)dg) >> 6);  // fewer than 64 each
    bad |= (u32)((u64)P >> 32) ^ (u32)((int)P >> 31);                                 // priority in int32
    bad |= (u32)K >> 31;
    // 2 <= T < 2^26, 1 <= D <= T
    ok &= (u32)T - 2u < kFastLimit - 2u && (u32)D - 1u < (u32)T;
    prio[s] = (int)P;
    uses_gpu[s] = lane + 32 * s < n && (u32)dg > 0;
  }
  // (every task has 0 .. 63 segments of a kind and the last one ends where the slice does: so all
  // offsets lie inside the staged slices)
  const u32 c_first = (u32)(u64)sCo[0], g_first = (u32)(u64)sGo[0];
  ok &= (u32)sCo[n] - c_first == ((me.packed >> 9) & 0x7ffu) && (u32)sGo[n] - g_first == ng;
  // ---- ... and of the segment values: the three slices lie side by side --------------------------
  {
    u32 lo = 0;
    const u32 from = (off1.z & ~15u) + 16u * (u32)lane, to = off2.y;
#pragma unroll 4
    for (u32 e = from; e < to; e += 512u) {
      const uint4 v = *reinterpret_cast<const uint4 *>(stage + e);
      bad |= v.y | v.w, lo |= v.x | v.z;
    }
    bad |= lo >> 26;
  }
  // ---- order: rank by (priority desc, position asc) ---------------------------------------------
  int pmax = prio[0];
#pragma unroll
  for (int s = 1; s < SLOTS; ++s) pmax = prio[s] > pmax ? prio[s] : pmax;
  pmax = __reduce_max_sync(kFull, pmax);
  bool dense = true;  // distinct priorities max-n+1 .. max: the rank is max - priority
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    rank[s] = (int)((u32)pmax - (u32)prio[s]);
    dense &= (u32)rank[s] < (u32)n;
  }
  if (__any_sync(kFull, bad != 0 || !ok)) {
    next();
    return kHeadUndecided;
  }
  dense = __all_sync(kFull, dense);
  if (dense) {
#pragma unroll
    for (int s = 0; s < SLOTS; ++s)
      w.pos_of_rank[rank[s]] = (unsigned char)(lane + 32 * s < n ? lane + 32 * s : n - 1);
    __syncwarp();
    bool uniq = true;
#pragma unroll
    for (int s = 0; s < SLOTS; ++s)
      uniq &= w.pos_of_rank[rank[s]] == (unsigned char)(lane + 32 * s < n ? lane + 32 * s : n - 1);
    dense = __all_sync(kFull, uniq);
  }
  if (!dense) {  // any priorities: count the tasks that come before
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) rank[s] = 0;
    for (int q = 0; q < n; ++q) {
      const int pq = (int)sP[q];
#pragma unroll
      for (int s = 0; s < SLOTS; ++s) rank[s] += (pq > prio[s] || (pq == prio[s] && q < lane + 32 * s)) ? 1 : 0;
    }
    __syncwarp();
#pragma unroll
    for (int s = 0; s < SLOTS; ++s)
      if (lane + 32 * s < n) w.pos_of_rank[rank[s]] = (unsigned char)(lane + 32 * s);
    __syncwarp();
  }
  int n_rt = n;  // best-effort tasks (flag set, priority <= 0) rank behind every real-time task
  if (best_effort) {
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) n_rt -= __popc(__ballot_sync(kFull, lane + 32 * s < n && prio[s] <= 0));
  }
  int n_gpu = 0;  // N_g
  if (!kGcaps) {
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) n_gpu += __popc(__ballot_sync(kFull, uses_gpu[s]));
  }
  // ---- the first ranks: two lanes add up the segments of one rank ---------------------------------
  const int limit = n_rt < kHeadRanks ? n_rt : kHeadRanks;
  const int r2 = lane >> 1, sub = lane & 1;
  const int pos = w.pos_of_rank[r2 < n ? r2 : 0];
  const u32 T = (u32)sT[pos], D = (u32)sD[pos], core = (u32)sK[pos];
  u32 A = 0, Ge = 0, slices = 0;
  const u32 c0 = (u32)sCo[pos] - c_first, cn = (u32)sCo[pos + 1] - c_first;
  const u32 g0 = (u32)sGo[pos] - g_first, gn = (u32)sGo[pos + 1] - g_first;
  {
    const i64 *const sC = reinterpret_cast<const i64 *>(stage + off1.z);
    const i64 *const sM = reinterpret_cast<const i64 *>(stage + off1.w);
    const i64 *const sE = reinterpret_cast<const i64 *>(stage + off2.x);
#pragma unroll 1
    for (u32 j = c0 + sub; j < cn; j += 2) A += (u32)sC[j];
#pragma unroll 1
    for (u32 j = g0 + sub; j < gn; j += 2) {
      const u32 e = (u32)sE[j];
      A += (u32)sM[j], Ge += e;
      if (!kGcaps) {  // Eq. 3: slices of the pure GPU part
        if (p.l_mode == 0) slices += __umulhi(e + (u32)p.L - 1u, p.l_magic) >> p.l_shift;
        else if (p.l_mode == 1) slices += e;
        else slices += e > 0 ? 1u : 0u;
      }
    }
  }
  // (a lane has added up to 64 values below 2^26, the sums fit 32 bits; with every partial sum below
  // 2^26 the rank's sums do too)
  const bool mine = r2 < limit;
  bool wide = mine && ((A | Ge) >> 26) != 0;
  __syncwarp();
  next();  // nothing below reads the stage
  A += __shfl_xor_sync(kFull, A, 1), Ge += __shfl_xor_sync(kFull, Ge, 1);
  if (!kGcaps) slices += __shfl_xor_sync(kFull, slices, 1);
  PairConsts pc;
  pc.ovh = (u32)p.ovh;
  pc.slot_cost = (u64)p.L + pc.ovh;
  const u32 eta = gn - g0;
  u32 S, base;
  own_cost<kGcaps>(pc, A, Ge, eta, slices, n_gpu, S, base);
  wide |= mine && (T >= kNarrowLimit || (A | Ge) >> 26 || (kGcaps && S >> 26));
  if (mine && sub == 0) {
    rows.a(r2) = make_uint4(D, core, 0u, 0u);
    rows.b(r2) = make_uint4(T, A, Ge | (eta > 0 ? kRowGpu : 0u), S);
    rows.base(r2) = base;
  }
  if (__any_sync(kFull, wide)) return kHeadUndecided;
  __syncwarp();
  int made = 0;
  const Outcome o = recurrence_narrow<32, 1, MODE, false>(rows, limit, n_gpu, pc, literal, lane, kFull, made);
  if (o.verdict == 0 && limit < n_rt) return kHeadUndecided;
  __syncwarp();
  // ---- results: converged ranks first, then the sentinels by position -----------------------------
  i64 *const out = p.out_wcrt + me.a;
  if (sub == 0 && r2 < o.n_done) out[pos] = (i64)rows.R(r2);
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    if (lane + 32 * s < n && rank[s] >= o.n_done)
      out[lane + 32 * s] = rank[s] >= n_rt ? (i64)GCAPS_WCRT_BEST_EFFORT
                                           : (rank[s] == o.n_done ? (i64)o.verdict : (i64)GCAPS_WCRT_SKIPPED);
  }
  if (lane == 0) p.out_sched[me.t] = o.verdict == 0 ? GCAPS_SCHED_YES : GCAPS_SCHED_NO;
  return kFastDone;
}

// The full pass over one taskset, from global memory.
template <int SLOTS, int MODE>
__device__ __forceinline__ void full_pass(const KParams &p, const Ahead me, bool fast_call, u32 *buf, int lane) {
  int how = kFastDeclined;
  if (fast_call && (me.packed >> 31) != 0) {
    prefetch_segments<32>(p, me, lane);
    how = analyse_fast<32, SLOTS, 1 << MODE>(p, true, (i64)me.t, me.a, (int)(me.packed & 0x1ffu), buf, lane, kFull);
  }
  __syncwarp();
  if (how != kFastDone)  // the exact path reads task_off again and validates everything itself
    analyse_taskset<32, 32 * SLOTS>(p, (i64)me.t, *reinterpret_cast<GroupSmem<32 * SLOTS> *>(buf), lane, kFull);
  __syncwarp();
}

// The steps of walk_staged_bin on the device.
template <int SLOTS, int MODE>
struct StagedSteps {
  typedef FastLayout<32, SLOTS> Lay;
  static constexpr int MAXN = 32 * SLOTS;
  const KParams &p;
  const SliceTable &tab;
  StagedWarp<SLOTS> &w;
  unsigned char *stage;
  u32 stage_bytes;
  int bin, lane;
  unsigned int start, count, chunk;
  bool fast_call;
  u32 phase;
  unsigned int asked;
  Ahead me;

  __device__ __forceinline__ unsigned int pull(unsigned int n) {
    ask(n);
    return answer();
  }
  __device__ __forceinline__ void ask(unsigned int n) {
    asked = 0;
    if (lane == 0) asked = atomicAdd(&p.hdr->next[bin], n);
  }
  __device__ __forceinline__ unsigned int answer() { return __shfl_sync(kFull, asked, 0); }
  // lanes 0..chunk-1 each look up one taskset
  __device__ __forceinline__ void look_up(unsigned int first, int half) {
    if ((unsigned int)lane < chunk)
      w.ahead[half * kStagedChunk + lane] =
          look_up_taskset<MAXN, Lay::CAP>(p, first + lane < count ? p.perm[start + first + lane] : kNoTaskset);
    __syncwarp();
  }
  __device__ __forceinline__ void take(int half, int place) { me = w.ahead[half * kStagedChunk + place]; }
  __device__ __forceinline__ bool start_copies(int half, int place) {
    const Ahead &coming = w.ahead[half * kStagedChunk + place];
    return (coming.packed >> 31) != 0 && stage_taskset<SLOTS>(tab, coming, w, stage, stage_bytes, lane);
  }
  __device__ __forceinline__ bool wait() {
    const bool arrived = __all_sync(kFull, barrier_wait(&w.barrier, phase));
    if (arrived) phase ^= 1u;
    return arrived;
  }
  template <class Next>
  __device__ __forceinline__ bool head(Next next) {
    const int how = staged_head<SLOTS, MODE>(p, me, w, stage, lane, next);
    __syncwarp();
    return how == kFastDone;
  }
  __device__ __forceinline__ void first_try(bool decided) {
    if (lane == 0) atomicAdd(&p.hdr->first_tries[bin], decided ? 1u : 0x10001u);  // undecided | all
  }
  __device__ __forceinline__ bool most_undecided() const {
    const unsigned int tries = __ldcg(&p.hdr->first_tries[bin]);
    return (tries & 0xffffu) >= 32 && 4 * (tries >> 16) >= 3 * (tries & 0xffffu);
  }
  __device__ __forceinline__ void keep(int k, unsigned int entry) {
    if (lane == 0) w.left[k] = entry;
  }
  // (this warp pulled the entries: no one else looks at them in this launch)
  __device__ __forceinline__ void mark(unsigned int first, unsigned int n) {
    if ((unsigned int)lane < n) p.perm[start + first + lane] |= kDeferred;
  }
  __device__ __forceinline__ void mark_kept(int k) {
    __syncwarp();
    mark(w.left[k], 1);
  }
  __device__ __forceinline__ void full_pass(int k) {
    __syncwarp();
    ::full_pass<SLOTS, MODE>(p, look_up_taskset<MAXN, Lay::CAP>(p, p.perm[start + w.left[k]]), fast_call,
                             reinterpret_cast<u32 *>(stage), lane);
  }
  __device__ __forceinline__ void marked(unsigned int n) {
    if (lane == 0) atomicAdd(&p.hdr->deferred[bin], n);
  }
};

// One size bin, worked through by all warps of a persistent launch, a warp per taskset.
template <int SLOTS, int MODE>
__device__ __forceinline__ void run_staged_bin(const KParams &p, int bin, u32 stage_bytes, StagedWarp<SLOTS> &w,
                                               unsigned char *stage, const SliceTable &tab) {
  const unsigned int count = p.hdr->bin_count[bin];
  if (count == 0) return;
  const int lane = threadIdx.x & 31;
  const unsigned int n_warps = gridDim.x * (kStagedThreads / 32);
  const unsigned int chunk = count >= 32 * n_warps ? kStagedChunk : (count >= 8 * n_warps ? 4 : 1);
  const bool fast_call = p.ovh < (1 << 20);
  if (lane == 0) barrier_init(&w.barrier);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  __syncwarp();
  StagedSteps<SLOTS, MODE> steps = {p, tab, w, stage, stage_bytes, bin, lane, p.hdr->bin_start[bin], count, chunk, fast_call, 0u, 0u, {}};
  walk_staged_bin(steps, count, chunk, fast_call);
}

// The tasksets of a bin that its first launch marked, a warp per taskset, without stages.  Such tasksets run
// their recurrence to the end, tens of microseconds each, so the launch has to end evenly: permutation entries
// are pulled from a counter, pairs of them where a quarter of the bin or more is marked, else a quarter of a
// warp's share.  (In shares of 16 entries 12,289 tasksets of 128 tasks, a third of them marked, gave 768 of
// 3,552 warps all the work: 386 -> 297 us, 25,000 of 80 tasks 354 -> 312 us.)  Only where a bin holds 64
// entries or more per warp and few are marked does every warp look through its own share, 16 at a time.
// The next entries are looked up before the current ones are worked on.
template <int SLOTS, int MODE>
__device__ __forceinline__ void run_deferred_bin(const KParams &p, int bin, u32 *buf, Ahead *ahead) {
  typedef FastLayout<32, SLOTS> Lay;
  constexpr int MAXN = 32 * SLOTS;
  static_assert(sizeof(GroupSmem<MAXN>) <= sizeof(u32) * Lay::kWords, "exact path fits");
  const int lane = threadIdx.x & 31;
  const unsigned int start = p.hdr->bin_start[bin], count = p.hdr->bin_count[bin];
  const unsigned int marked = count > 0 ? __ldcg(&p.hdr->deferred[bin]) : 0;
  if (marked == 0) return;
  const bool fast_call = p.ovh < (1 << 20);
  const unsigned int n_warps = gridDim.x * (kBlockThreads / 32);
  const bool pulled = marked >= count / 4 || count < 64 * n_warps;
  unsigned int step = kMaxAhead;
  if (marked >= count / 4) step = 2;
  else if (pulled) step = count / (4 * n_warps) < 1 ? 1 : count / (4 * n_warps);
  unsigned int window = (blockIdx.x * (kBlockThreads / 32) + (threadIdx.x >> 5)) * step;  // (!pulled)
  int in_chunk = 0, which = 0;
  for (;;) {
    // the next entries
    unsigned int first = window;
    if (pulled) {
      if (lane == 0) first = atomicAdd(&p.hdr->next2[bin], step);
      first = __shfl_sync(kFull, first, 0);
    }
    window += n_warps * step;
    u32 t = 0;
    if (first < count && (unsigned int)lane < step && first + lane < count) t = __ldcg(&p.perm[start + first + lane]);
    const unsigned int found = __ballot_sync(kFull, (t & kDeferred) != 0);
    if (t & kDeferred)
      ahead[(which ^ 1) * kMaxAhead + __popc(found & ((1u << lane) - 1u))] = look_up_taskset<MAXN, Lay::CAP>(p, t & ~kDeferred);
    __syncwarp();
#pragma unroll 1
    for (int c = 0; c < in_chunk; ++c) full_pass<SLOTS, MODE>(p, ahead[which * kMaxAhead + c], fast_call, buf, lane);
    if (first >= count) break;
    in_chunk = __popc(found);
    which ^= 1;
  }
}

}  // namespace
#endif  // GCAPS_RTA_STAGED_CUH_
