// gcaps_igen.cu -- on-device generation of synthetic tasksets (the generation procedure of
// GCAPS, ECRTS 2024, arXiv 2406.05221, Sec. 7.1 / Table 3) for NVIDIA B200 (sm_100a).
//
// The generator itself is igen.h (integer-only; the host generator compiles the same
// definition).  gcaps_gen_count: one warp per taskset (for many small ones a thread) does what igen_begin
// defines (lane = task; the random source is counter-based, so every draw's position is known without the ones before it),
// writes the three sizes of the taskset and leaves what it drew per task (period, execution demand,
// priority, core, GPU segments: 12 bytes per task) and the position of the
// random stream in the workspace; three exclusive scans turn the sizes into offsets (block sums,
// one block over the block sums, block-local scan).  gcaps_gen_fill: one warp per taskset, lane =
// task; the random draws of a task start at a position that is a prefix sum over the tasks
// before it (the random source is counter-based).  The segments of 32 tasks at a time are split with
// lane = segment: random weights, quotients and stores all run over the segments side by side, and
// only the two sums of a task (its weights, its shares) are added up by the task's lane.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include "igen.h"
#include "rta_common.cuh"

using namespace gcaps_detail;

static_assert(sizeof(gcaps_gen_params_t) == sizeof(igen_params_t), "same layout");

namespace {

constexpr int kGenThreads = 128;
constexpr int kScanThreads = 256;
constexpr int kScanItems = 4 * kScanThreads;  // elements of one scan block

// workspace: off[3][count + 1] (tasks, CPU segments, GPU segments), block sums [3][blocks], then
// the per-taskset state: state_stride 32-bit words each -- key and counter of the random stream
// (4 words), then per task T, E and (priority | core << 16 | GPU segments << 24)
struct GenSpace {
  i64 *off[3];
  i64 *block_sum[3];
  i64 n_blocks;
  u32 *state;
  i64 state_stride;
};

__host__ __device__ inline i64 max_tasks_of(const igen_params_t &p) {
  const i64 m = (i64)p.cores_hi * (i64)p.tpc_hi;
  return m > IGEN_MAX_TASKS ? IGEN_MAX_TASKS : m;
}

__host__ __device__ inline i64 scan_blocks(i64 count) { return (count + kScanItems - 1) / kScanItems; }

// ---- the per-task part of the generator, a warp per taskset -----------------------------------------
struct CountTables {
  igen_exp2_tables_t exp2;
  uint64_t inverse[IGEN_MAX_TASKS + 1];  // floor((2^64 - 1) / d)
};

// Shared memory of one warp of the count kernel.
struct CountWarp {
  union {
    struct {
      u32 cut[IGEN_MAX_TASKS];  // by task: cut points of its core's utilisation as drawn, then its utilisation
      union {
        u32 sorted[IGEN_MAX_TASKS];  // the cut points in ascending order
        int writer[IGEN_MAX_TASKS];  // the draw of GPU-using tasks, see below
        __align__(16) u32 key[IGEN_MAX_TASKS];  // (T << 8 | position), for the ranks
      };
    };
    uint64_t load[IGEN_MAX_TASKS];  // worst fit: E / T in Q32
  };
  u32 T[IGEN_MAX_TASKS];
  short last[IGEN_MAX_TASKS], from[IGEN_MAX_TASKS];
  unsigned char core[IGEN_MAX_TASKS], eta[IGEN_MAX_TASKS];
  u32 start[IGEN_MAX_CORES + 1];  // first task of a core
  u32 ctr[IGEN_MAX_CORES];        // draws in front of a core's
  u32 util[IGEN_MAX_CORES];       // utilisation of a core, Q32
  u32 pad_[3];
};
static_assert(sizeof(CountWarp) % 16 == 0, "16-byte rows");

__device__ __forceinline__ uint64_t draw_at(uint64_t key, u32 position) {  // the position-th draw, from 1 on
  igen_rng_t r;
  r.key = key, r.ctr = position - 1;
  return igen_u64(&r);
}

// x mod d with inverse = floor((2^64 - 1) / d): the quotient umulhi(x, inverse) is at most one too small
__device__ __forceinline__ u32 mod_by(uint64_t x, u32 d, uint64_t inverse) {
  const u32 r = (u32)x - (u32)__umul64hi(x, inverse) * d;  // below 2 d
  return r >= d ? r - d : r;
}
// igen_int of the draw x; `inverse`: that of hi - lo + 1 (0 for hi <= lo)
__device__ __forceinline__ int int_from(uint64_t x, int lo, int hi, uint64_t inverse) {
  return hi <= lo ? lo : lo + (int)mod_by(x, (u32)(hi - lo) + 1u, inverse);
}
// What the count kernel needs of the parameters beside them.
struct CountConsts {
  uint64_t inv_cores, inv_tpc, inv_seg;  // of the three ranges of integers
  u32 bucket_shift, bucket_first;        // periods (below 2^24) lie in up to 256 buckets by the leading bits of their floating-point form
};
inline CountConsts count_consts(const igen_params_t &p) {
  auto inverse = [](int lo, int hi) -> uint64_t { return hi <= lo ? 0 : ~0ULL / ((uint64_t)(hi - lo) + 1); };
  auto bits = [](i64 period) -> u32 {
    const float f = (float)period;
    u32 b;
    memcpy(&b, &f, sizeof(b));
    return b;
  };
  CountConsts c;
  c.inv_cores = inverse(p.cores_lo, p.cores_hi), c.inv_tpc = inverse(p.tpc_lo, p.tpc_hi);
  c.inv_seg = inverse(p.gpu_mode == 0 && p.seg_lo < 1 ? 1 : p.seg_lo, p.seg_hi);
  c.bucket_shift = 0;
  while ((bits(p.period_hi) >> c.bucket_shift) - (bits(p.period_lo) >> c.bucket_shift) > 255u) c.bucket_shift += 1;
  c.bucket_first = bits(p.period_lo) >> c.bucket_shift;
  return c;
}
__device__ __forceinline__ uint64_t range_from(uint64_t x, uint64_t lo, uint64_t hi) {  // igen_range of the draw x
  return hi <= lo ? lo : lo + igen_mul_shr32(hi - lo, x >> 32);
}

// A thread per taskset, step by step as igen.h says.  For many small tasksets, where most lanes of a warp per
// taskset would have no task (see thread_per_taskset).
__global__ void __launch_bounds__(kGenThreads) gen_count_thread_kernel(igen_params_t p, i64 first, i64 count, GenSpace w) {
  const i64 t = (i64)blockIdx.x * kGenThreads + threadIdx.x;
  if (t >= count) return;
  igen_state_t s;
  igen_begin(&p, (uint64_t)(first + t), &s);
  w.off[0][t] = s.n, w.off[1][t] = s.n_csegs, w.off[2][t] = s.n_gsegs;
  u32 *st = w.state + t * w.state_stride;
  st[0] = (u32)s.rng.key, st[1] = (u32)(s.rng.key >> 32);
  st[2] = (u32)s.rng.ctr, st[3] = (u32)(s.rng.ctr >> 32);
  for (int i = 0; i < s.n; ++i) {
    st[4 + 3 * i] = s.T[i];
    st[5 + 3 * i] = s.E[i];
    st[6 + 3 * i] = (u32)s.prio[i] | ((u32)s.core[i] << 16) | ((u32)s.eta[i] << 24);
  }
}

// A thread's chain through a taskset grows with the square of its n tasks; the throughput of a thread per
// taskset is up to 1.6 times (8 tasks) that of a warp per taskset, and beyond 48 tasks it is less.  The two take the
// same time at 100 n^2 to 300 n^2 tasksets: with the fill pass 160 n^2 tasksets of 8 / 16 / 24 / 32 / 40 / 48 tasks 106 / 167 /
// 301 / 569 / 1,110 / 1,771 us (threads / warps: 111 / 179 / 325 / 530 / 1,139 / 1,760), 40 n^2 of them 104 / 124 / 165 / 246 /
// 397 / 571 by threads and 103 / 113 / 139 / 192 / 340 / 498 by warps; 64 tasks are faster by warps at every count
// (1,500,000: 8.39 / 7.45 ms).
inline bool thread_per_taskset(const igen_params_t &p, i64 count) {
  const i64 n = max_tasks_of(p);
  return n <= 48 && count >= 160 * n * n;
}

// Bound by instruction issue.  2^y by two looked-up factors instead of fourteen conditional ones, remainders by
// reciprocals and ranks by buckets instead of comparing all pairs: 250,000 `large` tasksets 1.20 -> 0.90 ms.  A thread
// per taskset took 1.40 ms (2.3 KB of state per thread in local memory).
__global__ void __launch_bounds__(kGenThreads) gen_count_kernel(igen_params_t p, CountConsts consts, int most_tasks, i64 first,
                                                                 i64 count, GenSpace w) {
  __shared__ CountWarp warps[kGenThreads / 32];
  __shared__ CountTables table;
  CountWarp &s = warps[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  constexpr int kEntries = (1 << IGEN_LEAD_BITS) + 2 * (1 << IGEN_TAIL_BITS);
#pragma unroll 1
  for (int e = threadIdx.x; e < kEntries; e += kGenThreads) igen_exp2_entry(&table.exp2, e);
  for (int d = threadIdx.x + 1; d <= most_tasks; d += kGenThreads) table.inverse[d] = ~0ULL / (uint64_t)d;
  const int seg_lo = p.gpu_mode == 0 && p.seg_lo < 1 ? 1 : p.seg_lo;
  __syncthreads();
#pragma unroll 1
  for (i64 t = (i64)blockIdx.x * (kGenThreads / 32) + (threadIdx.x >> 5); t < count; t += (i64)gridDim.x * (kGenThreads / 32)) {
    igen_rng_t rng;
    igen_rng_init(&rng, p.seed, p.stream, (uint64_t)(first + t));
    const uint64_t key = rng.key;
    int cores = int_from(draw_at(key, 1), p.cores_lo, p.cores_hi, consts.inv_cores);
    if (cores > IGEN_MAX_CORES) cores = IGEN_MAX_CORES;
    const bool harmonic = (draw_at(key, 2) >> 32) < p.harmonic;
    u32 ctr = 2;  // draws so far
    int n = 0;
    // tasks per core: a core takes a draw for its tasks, one for its utilisation, one per cut point
#pragma unroll 1
    for (int c = 0; c < cores; ++c) {
      int m = p.tpc_hi <= p.tpc_lo ? p.tpc_lo : int_from(draw_at(key, ctr + 1), p.tpc_lo, p.tpc_hi, consts.inv_tpc);
      if (n + m > IGEN_MAX_TASKS) m = IGEN_MAX_TASKS - n;
      if (lane == 0) s.start[c] = (u32)n, s.ctr[c] = ctr;
      for (int k = lane; k < m; k += 32) s.core[n + k] = (unsigned char)c;
      ctr += 2 + (m > 1 ? m - 1 : 0);
      n += m;
    }
    if (lane == 0) s.start[cores] = (u32)n;
    __syncwarp();
    for (int c = lane; c < cores; c += 32) s.util[c] = (u32)range_from(draw_at(key, s.ctr[c] + 2), p.util_lo, p.util_hi);
#pragma unroll 1
    for (int i = lane; i < n; i += 32) {
      const int c = s.core[i], k = i - (int)s.start[c];
      if (i + 1 < (int)s.start[c + 1]) s.cut[i] = (u32)(draw_at(key, s.ctr[c] + 3 + k) >> 32);
      s.eta[i] = 0, s.last[i] = -1;
    }
    __syncwarp();
#pragma unroll 1
    for (int i = lane; i < n; i += 32) {  // the cut points of a core in ascending order
      const int c = s.core[i], from = (int)s.start[c], last = (int)s.start[c + 1] - 1;
      if (i < last) {
        const u32 x = s.cut[i];
        int r = from;
#pragma unroll 1
        for (int q = from; q < last; ++q) {
          const u32 y = s.cut[q];
          r += (y < x || (y == x && q < i)) ? 1 : 0;
        }
        s.sorted[r] = x;
      }
    }
    __syncwarp();
#pragma unroll 1
    for (int i = lane; i < n; i += 32) {  // a task's share of its core (the last one takes what is left)
      const int c = s.core[i], from = (int)s.start[c], last = (int)s.start[c + 1] - 1;
      if (i < last) s.cut[i] = (u32)(((uint64_t)s.util[c] * (s.sorted[i] - (i > from ? s.sorted[i - 1] : 0u))) >> 32);
    }
    __syncwarp();
#pragma unroll 1
    for (int i = lane; i < n; i += 32) {
      const int c = s.core[i], from = (int)s.start[c], last = (int)s.start[c + 1] - 1;
      if (i == last) {
        u32 left = s.util[c];
#pragma unroll 1
        for (int q = from; q < last; ++q) left -= s.cut[q];
        s.cut[i] = left;
      }
    }
    // periods
#pragma unroll 1
    for (int i = lane; i < n; i += 32) {
      i64 T;
      if (harmonic) {
        const i64 T0 = (i64)igen_exp2_by(&table.exp2, range_from(draw_at(key, ctr + 1 + 2 * i), p.log2_lo, p.log2_hi0));
        T = T0 << int_from(draw_at(key, ctr + 2 + 2 * i), 0, 10, ~0ULL / 11);
      } else {
        T = (i64)igen_exp2_by(&table.exp2, range_from(draw_at(key, ctr + 1 + i), p.log2_lo, p.log2_hi));
      }
      if (T < p.period_lo) T = p.period_lo;
      if (T > p.period_hi) T = p.period_hi;
      s.T[i] = (u32)T;
    }
    ctr += harmonic ? 2 * n : n;
    // which tasks use the GPU, and how many segments they ask for
    if (p.gpu_mode == 0) {
      // A partial Fisher-Yates shuffle of 0 .. n-1: step k swaps positions k and j_k >= k, and the task
      // then at position k is drawn.  Position k is last written, before step k, by the largest k' < k
      // with j_k' = k (`writer`), and then holds what was at position k' before step k': following the
      // writers to the end gives the task (v).  What step k draws was at position j_k: v of the last
      // k' < k with the same j, or j_k itself.
      int ng = (int)((p.gpu_frac * (uint64_t)n + (1ULL << 31)) >> 32);
      if (ng > n) ng = n;
      for (int i = lane; i < n; i += 32) s.writer[i] = -1;
      __syncwarp();
#pragma unroll 1
      for (int k0 = 0; k0 < ng; k0 += 32) {
        const int k = k0 + lane;
        const int j = k < ng ? k + (int)mod_by(draw_at(key, ctr + 1 + 2 * k), (u32)(n - k), table.inverse[n - k]) : -1 - lane;
        const u32 same = __match_any_sync(kFull, j);
        const u32 below = same & ((1u << lane) - 1u);
        int before = -1;
        if (k < ng) {
          before = below ? k0 + 31 - __clz((int)below) : (int)s.last[j];
          if (j != k) atomicMax(&s.writer[j], k);
        }
        __syncwarp();
        if (k < ng) {
          if ((same >> lane) == 1u) s.last[j] = (short)k;  // the last of its kind in this round
          s.from[k] = (short)(before >= 0 ? before : ~j);   // a step to follow, or ~task
        }
        __syncwarp();
      }
#pragma unroll 1
      for (int k = lane; k < ng; k += 32) {
        int task = s.from[k];
        if (task >= 0) {
          while (s.writer[task] >= 0) task = s.writer[task];
        } else {
          task = ~task;
        }
        s.eta[task] = (unsigned char)int_from(draw_at(key, ctr + 2 + 2 * k), seg_lo, p.seg_hi, consts.inv_seg);
      }
      ctr += 2 * ng;
    } else {
#pragma unroll 1
      for (int i = lane; i < n; i += 32) s.eta[i] = (unsigned char)int_from(draw_at(key, ctr + 1 + i), p.seg_lo, p.seg_hi, consts.inv_seg);
      ctr += n;
    }
    __syncwarp();
    // execution demand; a task drops segments until every one gets at least 1 us
    u32 *st = w.state + t * w.state_stride;
    u32 nc = 0, ngs = 0;
#pragma unroll 1
    for (int i = lane; i < n; i += 32) {
      const u32 T = s.T[i];
      uint64_t E = ((uint64_t)s.cut[i] * T + (1ULL << 31)) >> 32;
      if (E < 1) E = 1;
      if (E > T) E = T;
      u32 eta = s.eta[i] > IGEN_MAX_SEGS ? IGEN_MAX_SEGS : s.eta[i];
      if (eta > ((u32)E - 1) / 2) eta = ((u32)E - 1) / 2;
      s.eta[i] = (unsigned char)eta;
      nc += eta + 1, ngs += eta;
      st[4 + 3 * i] = T, st[5 + 3 * i] = (u32)E;
    }
    __syncwarp();
    if (p.wfd) {
      // worst fit, decreasing by utilisation (ties: lower index first): the order by counting, then one
      // task after the other to the core with the least load (lane: cores lane and lane + 32)
#pragma unroll 1
      for (int i = lane; i < n; i += 32) s.load[i] = ((uint64_t)st[5 + 3 * i] << 32) / s.T[i];
      __syncwarp();
#pragma unroll 1
      for (int i = lane; i < n; i += 32) {
        const uint64_t u = s.load[i];
        int r = 0;
#pragma unroll 1
        for (int q = 0; q < n; ++q) {
          const uint64_t y = s.load[q];
          r += (y > u || (y == u && q < i)) ? 1 : 0;
        }
        s.from[r] = (short)i;
      }
      __syncwarp();
      uint64_t load0 = lane < cores ? 0 : ~0ULL >> 8, load1 = lane + 32 < cores ? 0 : ~0ULL >> 8;
#pragma unroll 1
      for (int k = 0; k < n; ++k) {
        const int i = s.from[k];
        // least (load, core): loads stay below 2^41, in two halves with the core behind the lower one
        const bool second = load1 < load0;
        const uint64_t mine = second ? load1 : load0;
        const u32 hi = mine >= (1ULL << 48) ? 0xffffffffu : (u32)(mine >> 20);
        const u32 least = __reduce_min_sync(kFull, hi);
        const u32 lo = hi == least ? (((u32)mine & 0xfffffu) << 6) | (u32)(second ? lane + 32 : lane) : 0xffffffffu;
        const u32 best = __reduce_min_sync(kFull, lo) & 63u;
        if ((best & 31u) == (u32)lane) {
          if (best >= 32) load1 += s.load[i];
          else load0 += s.load[i];
        }
        if (lane == 0) s.core[i] = (unsigned char)best;
      }
      __syncwarp();
    }
    // rate-monotonic priorities: shorter period = higher, ties by position.  Periods below 2^24 with the
    // position behind them are distinct 32-bit keys.  Log-uniform as they are, the leading bits of their
    // floating-point form spread them evenly over 256 buckets, as narrow as their range allows; a key's rank is its
    // bucket's start and the smaller keys in the bucket, which are compared four at a time as equal periods share one.
    // 100,000 tasksets of 80 tasks, one key at a time (comparing all pairs) -> this: equal periods 608 (487) -> 468 us, 100,000
    // to 100,500 us 547 (501) -> 376, harmonic ones 547 (514) -> 458, 1 ms to 1 s 372 (501) -> 376.
    if (p.period_hi < (1LL << 24)) {
      for (int c = lane; c < 64; c += 32) reinterpret_cast<uint4 *>(s.cut)[c] = make_uint4(0, 0, 0, 0);
      __syncwarp();
      auto bucket = [&](u32 T) -> u32 { return (__float_as_uint((float)T) >> consts.bucket_shift) - consts.bucket_first; };
#pragma unroll 1
      for (int i = lane; i < n; i += 32) s.from[i] = (short)atomicAdd(&s.cut[bucket(s.T[i])], 1u);
      __syncwarp();
      {  // starts of the buckets, eight per lane
        uint4 x = reinterpret_cast<uint4 *>(s.cut)[2 * lane], y = reinterpret_cast<uint4 *>(s.cut)[2 * lane + 1];
        x.y += x.x, x.z += x.y, x.w += x.z, y.x += x.w, y.y += y.x, y.z += y.y, y.w += y.z;
        u32 before = y.w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const u32 o = __shfl_up_sync(kFull, before, d);
          if (lane >= d) before += o;
        }
        before -= y.w;
        reinterpret_cast<uint4 *>(s.cut)[2 * lane] = make_uint4(before, before + x.x, before + x.y, before + x.z);
        reinterpret_cast<uint4 *>(s.cut)[2 * lane + 1] = make_uint4(before + x.w, before + y.x, before + y.y, before + y.z);
      }
      __syncwarp();
#pragma unroll 1
      for (int i = lane; i < n; i += 32) s.key[s.cut[bucket(s.T[i])] + (u32)s.from[i]] = (s.T[i] << 8) | (u32)i;
      if (lane < (-n & 3)) s.key[n + lane] = 0xffffffffu;
      __syncwarp();
#pragma unroll 1
      for (int i = lane; i < n; i += 32) {
        const u32 T = s.T[i], c = bucket(T), mine = (T << 8) | (u32)i;
        const u32 to = c < 255 ? s.cut[c + 1] : (u32)n;
        // four keys at a time: those in front of the bucket are smaller, those behind it are not
        u32 higher = s.cut[c] & ~3u;
#pragma unroll 1
        for (u32 q = higher; q < to; q += 4) {
          const uint4 y = *reinterpret_cast<const uint4 *>(&s.key[q]);
          higher += (y.x < mine ? 1u : 0u) + (y.y < mine ? 1u : 0u) + (y.z < mine ? 1u : 0u) + (y.w < mine ? 1u : 0u);
        }
        st[6 + 3 * i] = ((u32)n - higher) | ((u32)s.core[i] << 16) | ((u32)s.eta[i] << 24);
      }
    } else {
#pragma unroll 1
      for (int i = lane; i < n; i += 32) {
        int higher = 0;
        const u32 T = s.T[i];
#pragma unroll 1
        for (int q = 0; q < n; ++q) higher += s.T[q] < T + (q < i ? 1u : 0u) ? 1 : 0;
        st[6 + 3 * i] = (u32)(n - higher) | ((u32)s.core[i] << 16) | ((u32)s.eta[i] << 24);
      }
    }
    nc = __reduce_add_sync(kFull, nc), ngs = __reduce_add_sync(kFull, ngs);
    if (lane == 0) {
      w.off[0][t] = n, w.off[1][t] = nc, w.off[2][t] = ngs;
      st[0] = (u32)key, st[1] = (u32)(key >> 32), st[2] = ctr, st[3] = 0;
    }
    __syncwarp();
  }
}

__device__ __forceinline__ i64 block_exclusive_scan(i64 v, i64 *total, i64 *warp_sums) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  i64 x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const i64 y = __shfl_up_sync(kFull, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) warp_sums[warp] = x;
  __syncthreads();
  if (warp == 0) {
    i64 ws = lane < kScanThreads / 32 ? warp_sums[lane] : 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const i64 y = __shfl_up_sync(kFull, ws, d);
      if (lane >= d) ws += y;
    }
    if (lane < kScanThreads / 32) warp_sums[lane] = ws;  // inclusive sums of the warps
  }
  __syncthreads();
  const i64 before = warp > 0 ? warp_sums[warp - 1] : 0;
  *total = warp_sums[kScanThreads / 32 - 1];
  __syncthreads();
  return before + x - v;
}

// sums of every block of kScanItems sizes, for the three arrays (blockIdx.y)
__global__ void __launch_bounds__(kScanThreads) scan_sums_kernel(GenSpace w, i64 count) {
  __shared__ i64 warp_sums[kScanThreads / 32];
  const i64 *in = w.off[blockIdx.y];
  const i64 base = (i64)blockIdx.x * kScanItems + 4 * threadIdx.x;
  i64 v = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (base + j < count) v += in[base + j];
  i64 total;
  block_exclusive_scan(v, &total, warp_sums);
  if (threadIdx.x == 0) w.block_sum[blockIdx.y][blockIdx.x] = total;
}

// one block per array: block sums -> exclusive offsets of the blocks; the grand total goes to
// off[a][count] and to out_totals[a]
__global__ void __launch_bounds__(kScanThreads) scan_blocks_kernel(GenSpace w, i64 count, i64 *out_totals) {
  __shared__ i64 warp_sums[kScanThreads / 32];
  i64 *bs = w.block_sum[blockIdx.x];
  i64 carry = 0;
  for (i64 b0 = 0; b0 < w.n_blocks; b0 += kScanThreads) {
    const i64 b = b0 + threadIdx.x;
    const i64 v = b < w.n_blocks ? bs[b] : 0;
    i64 total;
    const i64 ex = block_exclusive_scan(v, &total, warp_sums);
    if (b < w.n_blocks) bs[b] = carry + ex;
    carry += total;
  }
  if (threadIdx.x == 0) {
    w.off[blockIdx.x][count] = carry;
    out_totals[blockIdx.x] = carry;
  }
}

// sizes -> exclusive offsets, in place
__global__ void __launch_bounds__(kScanThreads) scan_apply_kernel(GenSpace w, i64 count) {
  __shared__ i64 warp_sums[kScanThreads / 32];
  i64 *io = w.off[blockIdx.y];
  const i64 base = (i64)blockIdx.x * kScanItems + 4 * threadIdx.x;
  i64 x[4], v = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    x[j] = base + j < count ? io[base + j] : 0;
    v += x[j];
  }
  i64 total;
  i64 run = w.block_sum[blockIdx.y][blockIdx.x] + block_exclusive_scan(v, &total, warp_sums);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (base + j < count) io[base + j] = run;
    run += x[j];
  }
}

struct GenOut {
  i64 *task_off, *period, *deadline, *priority, *core, *cseg_off, *cseg_wcet, *gseg_off, *gseg_misc, *gseg_exec;
  i64 cap_tasks, cap_csegs, cap_gsegs;
};

__device__ __forceinline__ u32 warp_exclusive(u32 v, int lane, u32 *total) {
  u32 x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const u32 y = __shfl_up_sync(kFull, x, d);
    if (lane >= d) x += y;
  }
  *total = __shfl_sync(kFull, x, 31);
  return x - v;
}

constexpr int kFillParts = 32 * (IGEN_MAX_SEGS + 1);  // segments of a kind of 32 tasks, at most

// Shared memory of one warp of the fill kernel, for 32 tasks.
struct FillWarp {
  uint64_t weights[32];  // by task: sum of its weights (Q32)
  double inverse[32];    // ... and its reciprocal
  u32 spare[32];         // what is shared out beyond 1 us per segment
  u32 draw[32];          // position of the first weight's draw within the taskset's stream
  u32 share[kFillParts];  // by segment: the random fraction of its weight, then its share of `spare`
  unsigned short first[32];         // first segment of the task
  unsigned char owner[kFillParts];  // by segment: the task's lane
};

// Splits `total` us of this lane's task into `parts` segments (0: none) like igen_split does, the tasks
// of all lanes at once.  `draw`: position of the task's first weight.  The segments of the lanes lie one
// behind the other from out[0] on (this lane's from out[first] on, n_parts in all); FIFTH: a fifth of each goes to `fifth`.
//
// igen_split's quotient floor(spare * w / sum of weights) is taken in double precision with the task's
// reciprocal (good to 2^-45, so that a quotient below 2^31 is off by less than 2^-14 before it is rounded down, by at
// most 1 after) and settled by its remainder.
template <bool FIFTH>
__device__ __forceinline__ void split_tasks(FillWarp &w, uint64_t key, uint64_t ctr, u32 draw, u32 total, u32 parts,
                                            u32 first, u32 n_parts, i64 *out, i64 *fifth, int lane) {
  if (!__any_sync(kFull, parts > 1)) {  // a task's only segment takes all of it, whatever its weight
    if (parts > 0) {
      const u32 small = FIFTH ? total / 5u : 0u;
      out[first] = (i64)(total - small);
      if (FIFTH) fifth[first] = (i64)small;
    }
    return;
  }
  w.spare[lane] = total - parts;
  w.draw[lane] = draw;
  w.first[lane] = (unsigned short)first;
#pragma unroll 1
  for (u32 j = 0; j < parts; ++j) w.owner[first + j] = (unsigned char)lane;
  __syncwarp();
#pragma unroll 1
  for (u32 q = lane; q < n_parts; q += 32) {
    const int i = w.owner[q];
    igen_rng_t rng;
    rng.key = key, rng.ctr = ctr + w.draw[i] + (q - w.first[i]);
    w.share[q] = (u32)igen_unit(&rng);
  }
  __syncwarp();
  uint64_t sum = (uint64_t)parts << 32;
#pragma unroll 1
  for (u32 j = 0; j < parts; ++j) sum += w.share[first + j];
  w.weights[lane] = sum;
  {  // the reciprocal to 46 bits: one step of Newton's iteration from single precision
    const double d = (double)(sum + (parts == 0 ? 1 : 0)), r = (double)__frcp_rn((float)d);
    w.inverse[lane] = r * (2.0 - d * r);
  }
  __syncwarp();
#pragma unroll 1
  for (u32 q = lane; q < n_parts; q += 32) {
    const int i = w.owner[q];
    const u32 spare = w.spare[i], u = w.share[q];
    const uint64_t of = w.weights[i];
    u32 x = (u32)((double)spare * ((double)u + 4294967296.0) * w.inverse[i]);
    const i64 rem = (i64)(((uint64_t)spare << 32) + (uint64_t)spare * u - (uint64_t)x * of);
    if (rem < 0) x -= 1;
    else if ((uint64_t)rem >= of) x += 1;
    w.share[q] = x;
  }
  __syncwarp();
  if (parts > 0) {  // the last segment takes what is left
    u32 left = w.spare[lane];
#pragma unroll 1
    for (u32 j = 0; j + 1 < parts; ++j) left -= w.share[first + j];
    w.share[first + parts - 1] = left;
  }
  __syncwarp();
#pragma unroll 1
  for (u32 q = lane; q < n_parts; q += 32) {
    const u32 part = 1 + w.share[q], small = FIFTH ? part / 5u : 0u;
    out[q] = (i64)(part - small);
    if (FIFTH) fifth[q] = (i64)small;
  }
  __syncwarp();
}

// Bound by instruction issue and by the stores: 250,000 `large` tasksets (2.3 GB) 0.95 ms; a lane per
// task for everything took 1.43 ms (lanes wait for the task with the most segments, weights drawn
// twice, 8-byte stores far apart).  The GPU and the CPU parts of a round split side by side: no gain there, and 1,000,000
// tasksets of 8 tasks, whose GPU parts need no split, 1.03 -> 1.09 ms.
__global__ void __launch_bounds__(kGenThreads) gen_fill_kernel(igen_params_t p, i64 first, i64 count,
                                                                GenSpace w, GenOut o) {
  __shared__ FillWarp warps[kGenThreads / 32];
  FillWarp &mine_w = warps[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const i64 t = (i64)blockIdx.x * (kGenThreads / 32) + (threadIdx.x >> 5);
  if (t >= count) return;
  const i64 k0 = w.off[0][t], n = w.off[0][t + 1] - k0;
  const i64 c_start = w.off[1][t], g_start = w.off[2][t];
  if (lane == 0) o.task_off[t] = k0;
  const bool fits = k0 + n <= o.cap_tasks && w.off[1][t + 1] <= o.cap_csegs && w.off[2][t + 1] <= o.cap_gsegs;
  if (fits) {
    const u32 *st = w.state + t * w.state_stride;
    const uint64_t key = (uint64_t)st[0] | ((uint64_t)st[1] << 32);
    uint64_t ctr = (uint64_t)st[2] | ((uint64_t)st[3] << 32);
    u32 c_run = 0, g_run = 0;  // segments of the tasks before this round of 32
#pragma unroll 1
    for (i64 i0 = 0; i0 < n; i0 += 32) {
      const i64 i = i0 + lane;
      const bool mine = i < n;
      u32 T = 0, E = 0, pk = 0;
      if (mine) T = st[4 + 3 * i], E = st[5 + 3 * i], pk = st[6 + 3 * i];
      const u32 eta = pk >> 24, c_parts = mine ? eta + 1 : 0;
      u32 draws_total, c_total, g_total;
      const u32 draws_before = warp_exclusive(mine ? igen_task_draws((int)eta) : 0u, lane, &draws_total);
      const u32 c_before = warp_exclusive(c_parts, lane, &c_total);
      const u32 g_before = warp_exclusive(eta, lane, &g_total);
      // the draws of a task: the ratio, one weight per GPU segment, one per CPU segment
      igen_rng_t rng;
      rng.key = key, rng.ctr = ctr + draws_before;
      const u32 G = mine ? (u32)igen_task_gpu(&rng, (int64_t)E, (int)eta, p.ratio_lo, p.ratio_hi) : 0u;
      if (mine) {
        o.period[k0 + i] = T;
        o.deadline[k0 + i] = T;
        o.priority[k0 + i] = pk & 0xffffu;
        o.core[k0 + i] = (pk >> 16) & 0xffu;
        o.cseg_off[k0 + i] = c_start + c_run + c_before;
        o.gseg_off[k0 + i] = g_start + g_run + g_before;
      }
      split_tasks<true>(mine_w, key, ctr, draws_before + 1, G, eta, g_before, g_total, o.gseg_exec + g_start + g_run,
                        o.gseg_misc + g_start + g_run, lane);
      split_tasks<false>(mine_w, key, ctr, draws_before + 1 + eta, E - G, c_parts, c_before, c_total,
                         o.cseg_wcet + c_start + c_run, nullptr, lane);
      ctr += draws_total, c_run += c_total, g_run += g_total;
    }
  }
  if (t == count - 1 && lane == 0) {
    o.task_off[count] = w.off[0][count];
    if (w.off[0][count] <= o.cap_tasks) {
      o.cseg_off[w.off[0][count]] = w.off[1][count];
      o.gseg_off[w.off[0][count]] = w.off[2][count];
    }
  }
}

int g_count_blocks[64] = {0};

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

bool params_ok(const gcaps_gen_params_t *p) {
  return p && p->cores_lo >= 1 && p->cores_hi >= p->cores_lo && p->cores_hi <= IGEN_MAX_CORES &&
         p->tpc_lo >= 0 && p->tpc_hi >= p->tpc_lo && p->tpc_hi <= IGEN_MAX_TASKS &&
         p->util_lo <= p->util_hi && p->util_hi < (1ULL << 32) && p->log2_lo <= p->log2_hi &&
         p->log2_hi0 >= p->log2_lo && p->log2_hi < (31ULL << 32) && p->log2_hi0 < (31ULL << 32) &&
         p->period_lo >= 1 && p->period_hi >= p->period_lo && p->period_hi <= (1LL << 30) &&
         p->harmonic <= (1ULL << 32) && p->gpu_frac <= (1ULL << 32) && p->ratio_lo <= p->ratio_hi &&
         p->ratio_hi < (1ULL << 32) && (p->gpu_mode == 0 || p->gpu_mode == 1) && p->seg_lo >= 0 &&
         p->seg_hi >= p->seg_lo && p->seg_hi <= IGEN_MAX_SEGS;
}

int make_space(GenSpace *w, const gcaps_gen_params_t *params, int64_t count, void *workspace,
               size_t workspace_bytes) {
  if (!workspace || workspace_bytes < gcaps_gen_workspace_bytes(params, count) || ((uintptr_t)workspace & 255u))
    return GCAPS_ERR_WORKSPACE;
  unsigned char *b = (unsigned char *)workspace;
  const size_t off_bytes = align256((size_t)(count + 1) * sizeof(i64));
  w->n_blocks = scan_blocks(count);
  const size_t sum_bytes = align256((size_t)w->n_blocks * sizeof(i64));
  for (int a = 0; a < 3; ++a) {
    w->off[a] = (i64 *)(b + a * off_bytes);
    w->block_sum[a] = (i64 *)(b + 3 * off_bytes + a * sum_bytes);
  }
  igen_params_t p;
  memcpy(&p, params, sizeof(p));
  w->state = (u32 *)(b + 3 * off_bytes + 3 * sum_bytes);
  w->state_stride = 4 + 3 * max_tasks_of(p);
  return GCAPS_OK;
}

}  // namespace

extern "C" {

size_t gcaps_gen_workspace_bytes(const gcaps_gen_params_t *params, int64_t count) {
  if (count <= 0 || !params_ok(params)) return 0;
  igen_params_t p;
  memcpy(&p, params, sizeof(p));
  return 3 * align256((size_t)(count + 1) * sizeof(i64)) +
         3 * align256((size_t)scan_blocks(count) * sizeof(i64)) +
         align256((size_t)count * (size_t)(4 + 3 * max_tasks_of(p)) * sizeof(u32));
}

int gcaps_gen_count(const gcaps_gen_params_t *params, int64_t first, int64_t count,
                    int64_t *out_totals, void *workspace, size_t workspace_bytes, void *stream) {
  if (!params_ok(params) || first < 0 || count < 0 || count > 0x7fffffffLL || !out_totals)
    return GCAPS_ERR_INVALID_ARG;
  DeviceInfo di;
  int rc = device_info(&di);
  if (rc != GCAPS_OK) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  if (count == 0) {
    cudaError_t e = cudaMemsetAsync(out_totals, 0, 3 * sizeof(int64_t), st);
    if (e != cudaSuccess) {
      g_last_cuda_error = (int)e;
      return GCAPS_ERR_CUDA;
    }
    return GCAPS_OK;
  }
  GenSpace w;
  rc = make_space(&w, params, count, workspace, workspace_bytes);
  if (rc != GCAPS_OK) return rc;
  igen_params_t p;
  memcpy(&p, params, sizeof(p));
  constexpr int kWarps = kGenThreads / 32;
  cudaError_t e = cudaSuccess;
  if (thread_per_taskset(p, count)) {
    gen_count_thread_kernel<<<(unsigned int)((count + kGenThreads - 1) / kGenThreads), kGenThreads, 0, st>>>(
        p, (i64)first, (i64)count, w);
    e = cudaGetLastError();
  } else {
    int dev = 0;
    e = cudaGetDevice(&dev);
    // (once per device, before the number of resident blocks is looked up: as much shared memory as there is,
    // 24 instead of 16 warps per SM)
    if (e == cudaSuccess && __atomic_load_n(&g_count_blocks[dev & 63], __ATOMIC_ACQUIRE) == 0)
      e = cudaFuncSetAttribute(gen_count_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess)
      e = launch_persistent(gen_count_kernel, g_count_blocks, 0, (long long)((count + kWarps - 1) / kWarps), di.sm_count, st,
                            p, count_consts(p), (int)max_tasks_of(p), (i64)first, (i64)count, w);
  }
  if (e != cudaSuccess) {
    g_last_cuda_error = (int)e;
    return GCAPS_ERR_CUDA;
  }
  scan_sums_kernel<<<dim3((unsigned int)w.n_blocks, 3), kScanThreads, 0, st>>>(w, count);
  scan_blocks_kernel<<<3, kScanThreads, 0, st>>>(w, count, (i64 *)out_totals);
  scan_apply_kernel<<<dim3((unsigned int)w.n_blocks, 3), kScanThreads, 0, st>>>(w, count);
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    g_last_cuda_error = (int)e;
    return GCAPS_ERR_CUDA;
  }
  return GCAPS_OK;
}

int gcaps_gen_fill(const gcaps_gen_params_t *params, int64_t first, int64_t count,
                   const gcaps_tasksets_t *ts, void *workspace, size_t workspace_bytes, void *stream) {
  if (!params_ok(params) || first < 0 || count < 0 || count > 0x7fffffffLL || !ts) return GCAPS_ERR_INVALID_ARG;
  if (count == 0) return GCAPS_OK;
  if (!ts->task_off || ts->n_tasks < 0 || ts->n_csegs < 0 || ts->n_gsegs < 0 || !ts->cseg_off || !ts->gseg_off ||
      (ts->n_tasks > 0 && (!ts->period || !ts->deadline || !ts->priority || !ts->core)) ||
      (ts->n_csegs > 0 && !ts->cseg_wcet) || (ts->n_gsegs > 0 && (!ts->gseg_misc || !ts->gseg_exec)))
    return GCAPS_ERR_INVALID_ARG;
  DeviceInfo di;
  int rc = device_info(&di);
  if (rc != GCAPS_OK) return rc;
  GenSpace w;
  rc = make_space(&w, params, count, workspace, workspace_bytes);
  if (rc != GCAPS_OK) return rc;
  igen_params_t p;
  memcpy(&p, params, sizeof(p));
  GenOut o;
  o.task_off = (i64 *)ts->task_off, o.period = (i64 *)ts->period, o.deadline = (i64 *)ts->deadline;
  o.priority = (i64 *)ts->priority, o.core = (i64 *)ts->core, o.cseg_off = (i64 *)ts->cseg_off;
  o.cseg_wcet = (i64 *)ts->cseg_wcet, o.gseg_off = (i64 *)ts->gseg_off;
  o.gseg_misc = (i64 *)ts->gseg_misc, o.gseg_exec = (i64 *)ts->gseg_exec;
  o.cap_tasks = ts->n_tasks, o.cap_csegs = ts->n_csegs, o.cap_gsegs = ts->n_gsegs;
  constexpr int kWarps = kGenThreads / 32;
  gen_fill_kernel<<<(unsigned int)((count + kWarps - 1) / kWarps), kGenThreads, 0, (cudaStream_t)stream>>>(
      p, first, count, w, o);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    g_last_cuda_error = (int)e;
    return GCAPS_ERR_CUDA;
  }
  return GCAPS_OK;
}

}  // extern "C"
