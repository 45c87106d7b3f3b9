// rta_device.cuh -- device code of the analysis kernels, shared by the translation units that
// instantiate them: gcaps_rta.cu (one analysis per launch), gcaps_rta_direct.cu (small batches, a
// warp per taskset), gcaps_rta_sweep.cu and gcaps_rta_direct_sweep.cu (several analyses per launch).
// Batches of small tasksets of one size go through tiles (rta_tile.cuh, rta_tile_kept.cuh) and come
// here with what those leave over (gcaps_rta_rest.cu, gcaps_rta_rest_sweep.cu).  Internal.
//
// One warp analyses one taskset at a time:
//   stage      coalesced loads of the taskset's per-task slices into registers (lane = task)
//   aggregate  the per-task sums C_i, G^m_i, G^e_i: added up by the lane of the task, or (groups of
//              8 or 16 lanes with several tasks per lane) as differences of two running sums in
//              shared memory, as the RR slice count of Eq. 3 is
//   order      rank of every task by (priority desc, position asc); the per-task values move
//              through shared memory to the lane that owns the task's rank
//   iterate    for each task in rank order the recurrence of Eq. 1 with the lemma set of the
//              chosen analysis: lanes over the higher-priority interferers, each evaluating
//              ceil((R+J)/T_h)*W terms (division by the invariant T_h is a multiply-high by a
//              per-task reciprocal), summed across the warp
//   publish    the lane that owns the converged task keeps R_i and forms its jitters J^c, J^g
//   early exit the first deadline miss ends the taskset
//   write      out_wcrt (one value per task), out_sched (one byte per taskset)
// Loops with long bodies are kept rolled (#pragma unroll 1): unrolled by the compiler the code of one
// size bin was 120 KB instead of 56 KB, and instruction fetch was the largest stall wherever tasksets
// of a launch are at different places (four analyses of 100,001 20-task tasksets 773 -> 614 us, mixed
// sizes 1.45 -> 1.37 ms, 25 pairs of 200,000 tasksets 1.25 -> 1.07 ms, U/core 0.5 245 -> 226 us).
//
// The fast path holds every time in 32 bits and is taken when all values of a taskset are below
// 2^26 us; any other taskset goes through an exact 64-bit path with saturating arithmetic.
// Tasksets are binned by size (a small plan pass writes a permutation into the workspace) so that
// the warps of a launch hold the same number of tasks per lane; inside a launch warps pull chunks
// of tasksets from a counter, because iteration counts differ widely.
//
// A "one warp" above is a group of 8 or 16 lanes for tasksets of up to 32 tasks (two or four
// tasksets per warp).  gcaps_rta_multi_batch / gcaps_rta_sweep_batch use the same code with one
// staging, ordering and aggregation per taskset and one recurrence per requested analysis and
// (timeslice, overhead) pair.
#ifndef GCAPS_RTA_DEVICE_CUH_
#define GCAPS_RTA_DEVICE_CUH_

#include <cuda_runtime.h>
#include <stdint.h>

#include "rta_common.cuh"
#include "rta_recurrence.cuh"

namespace {

using namespace gcaps_detail;

// Shared-memory image of one taskset, indexed by priority rank unless noted.
template <int MAXN>
struct GroupSmem {
  u64 T[MAXN];     // period
  u64 D[MAXN];     // deadline
  u64 A[MAXN];     // C + G^m
  u64 Ge[MAXN];    // G^e
  u64 Star[MAXN];  // 2 * eps * eta^g   (GCAPS)   /   (L + theta) * slices, clamped   (RR)
  u64 R[MAXN];     // converged response time
  i64 prio_out[MAXN];  // by position: priority while ranking, then the output value
  int core[MAXN];
  int eta[MAXN];
  unsigned short ord[MAXN];  // rank -> position
};

// ---------------------------------------------------------------------------------------------
// the analysis of one taskset by a group of LPT lanes (exact 64-bit arithmetic)
// ---------------------------------------------------------------------------------------------
template <int LPT, int MAXN>
__device__ void analyse_taskset(const KParams &p, i64 t, GroupSmem<MAXN> &s, int lane,
                                unsigned int mask) {
  const int policy = p.policy & 0xff;
  const bool busy = (p.policy & GCAPS_RTA_BUSY) != 0;
  const bool literal = (p.policy & GCAPS_RTA_LITERAL) != 0;
  const bool best_effort = (p.policy & GCAPS_RTA_BEST_EFFORT) != 0;
  const u64 L = (u64)p.L, ovh = (u64)p.ovh;

  const i64 a = p.task_off[t] - p.task_base, b = p.task_off[t + 1] - p.task_base;
  if (a < 0 || b < a || b > p.n_tasks || b - a > MAXN) {
    // a range this launch cannot hold is a broken or oversized taskset: nothing is addressable
    if (lane == 0) p.out_sched[t] = GCAPS_SCHED_INVALID;
    return;
  }
  const int n = (int)(b - a);

  // ---- stage: priorities by position, domain check of the per-task scalars -------------------
  int bad = 0;
  for (int i = lane; i < n; i += LPT) {
    const i64 k = a + i;
    s.prio_out[i] = p.priority[k];
    const i64 T = p.period[k], D = p.deadline[k], c = p.core[k];
    if (T < 1 || T > GCAPS_RTA_MAX_TIME) bad |= GCAPS_BAD_PERIOD;
    if (D < 1 || D > T) bad |= GCAPS_BAD_DEADLINE;
    if (c < 0 || c > GCAPS_RTA_MAX_CORE) bad |= GCAPS_BAD_CORE;
  }
  __syncwarp(mask);

  // ---- order + aggregate: each lane ranks its tasks, sums their segments, stores by rank ------
  int n_gpu_lane = 0;
  for (int i = lane; i < n; i += LPT) {
    const i64 k = a + i;
    const i64 pi = s.prio_out[i];
    int rank = 0;
    for (int q = 0; q < n; ++q) {
      const i64 pq = s.prio_out[q];
      rank += (pq > pi || (pq == pi && q < i)) ? 1 : 0;
    }
    const i64 c0 = p.cseg_off[k] - p.cseg_base, c1 = p.cseg_off[k + 1] - p.cseg_base;
    const i64 g0 = p.gseg_off[k] - p.gseg_base, g1 = p.gseg_off[k + 1] - p.gseg_base;
    bool seg_ok = !(c0 < 0 || c1 < c0 || c1 > p.n_csegs || c1 - c0 > GCAPS_RTA_MAX_SEGMENTS ||
                    g0 < 0 || g1 < g0 || g1 > p.n_gsegs || g1 - g0 > GCAPS_RTA_MAX_SEGMENTS);
    u64 C = 0, Gm = 0, Ge = 0, slices = 0;
    if (seg_ok) {
      for (i64 j = c0; j < c1; ++j) {
        const i64 w = p.cseg_wcet[j];
        if (w < 0 || w > GCAPS_RTA_MAX_TIME) bad |= GCAPS_BAD_WCET;
        C += (u64)w;
      }
      for (i64 j = g0; j < g1; ++j) {
        const i64 m = p.gseg_misc[j], e = p.gseg_exec[j];
        if (m < 0 || m > GCAPS_RTA_MAX_TIME || e < 0 || e > GCAPS_RTA_MAX_TIME)
          bad |= GCAPS_BAD_WCET;
        Gm += (u64)m;
        Ge += (u64)e;
        if (policy == GCAPS_POLICY_RR && e > 0) slices += ceil_div64((u64)e, L);  // Eq. 3
      }
    } else {
      bad |= GCAPS_BAD_SEG_RANGE;
    }
    const int eta = seg_ok ? (int)(g1 - g0) : 0;
    n_gpu_lane += eta > 0 ? 1 : 0;
    s.T[rank] = (u64)p.period[k];
    s.D[rank] = (u64)p.deadline[k];
    s.A[rank] = C + Gm;
    s.Ge[rank] = Ge;
    s.Star[rank] = policy == GCAPS_POLICY_GCAPS ? 2 * ovh * (u64)eta : sat_mul(L + ovh, slices);
    s.core[rank] = (int)p.core[k];
    s.eta[rank] = eta;
    // a best-effort task (flag set, priority <= 0) ranks behind every real-time task; bit 15
    s.ord[rank] = (unsigned short)(i | ((best_effort && pi <= 0) ? 0x8000 : 0));
  }
  bad = group_or<LPT>(bad, mask);
  const int n_gpu = group_sum_int<LPT>(n_gpu_lane, mask);  // N_g
  __syncwarp(mask);
  if (bad) {
    if (p.out_wcrt)
      for (int i = lane; i < n; i += LPT) p.out_wcrt[a + i] = GCAPS_WCRT_INVALID;
    if (lane == 0) p.out_sched[t] = GCAPS_SCHED_INVALID;
    return;
  }
  for (int i = lane; i < n; i += LPT)
    s.prio_out[i] = (best_effort && s.prio_out[i] <= 0) ? GCAPS_WCRT_BEST_EFFORT : GCAPS_WCRT_SKIPPED;
  __syncwarp(mask);

  // ---- iterate: tasks in decreasing priority ---------------------------------------------------
  int sched = GCAPS_SCHED_YES;
  for (int pos = 0; pos < n; ++pos) {
    if (s.ord[pos] & 0x8000) break;  // only best-effort tasks from here on: nothing to bound
    const u64 Di = s.D[pos];
    const int core_i = s.core[pos];
    const bool gi = s.eta[pos] > 0;
    u64 base;
    u64 nu = 0;  // Lemma 4's interleaving-set size
    if (policy == GCAPS_POLICY_GCAPS) {
      // C_i + G*_i + B^C_i  (Sec. 6.3, Lemma 8); Star = 2*eps*eta
      base = s.A[pos] + s.Ge[pos] + s.Star[pos] + ((u64)s.eta[pos] + 1) * ovh;
    } else {
      // C_i + G_i + I^ie_i  (Lemma 1); Star = (L+theta)*slices
      base = s.A[pos] + s.Ge[pos] + (gi ? sat_mul(s.Star[pos], (u64)(n_gpu - 1)) : 0);
      if (busy) {
        int c = 0;
        for (int h = lane; h < pos; h += LPT) c += (s.core[h] == core_i && s.eta[h] > 0) ? 1 : 0;
        nu = (u64)(n_gpu - group_sum_int<LPT>(c, mask) + 1);
      }
    }
    u64 R = base;
    i64 verdict = 0;
    i64 sweeps = 0;
    for (;;) {
      if (R > Di) {
        verdict = GCAPS_WCRT_MISS;
        break;
      }
      if (sweeps >= GCAPS_RTA_ITER_CAP) {
        verdict = GCAPS_WCRT_ITER_LIMIT;
        break;
      }
      sweeps += 1;
      u64 part = 0;
      for (int h = lane; h < pos; h += LPT) {
        const u64 Th = s.T[h];
        const bool same = s.core[h] == core_i;
        const bool gh = s.eta[h] > 0;
        const u64 Rh = s.R[h];
        const u64 Jc = Rh - s.A[h], Jg = Rh - s.Ge[h];
        u64 term = 0;
        if (policy == GCAPS_POLICY_GCAPS && !busy) {
          if (same && !gh) term = sat_mul(ceil_div64(R, Th), s.A[h]);  // Lemma 15 (G^m_h = 0)
          if (same && gh) term = sat_mul(ceil_div64(R + Jc, Th), s.A[h] + s.Star[h]);
          if (same && gh && gi) term += sat_mul(ceil_div64(R + Jg, Th), s.Ge[h]);   // Lemma 13
          if (!same && gh && gi) term = sat_mul(ceil_div64(R + Jg, Th), s.Ge[h] + s.Star[h]);
        } else if (policy == GCAPS_POLICY_GCAPS) {
          if (same) {
            u64 W = s.A[h];                                                        // Lemma 12
            if (gh && (gi || !literal)) W += s.Ge[h] + s.Star[h];                  // Lemma 10
            term = sat_mul(ceil_div64(R, Th), W);
          } else if (gh) {
            term = sat_mul(ceil_div64(R + Jg, Th), s.Ge[h] + s.Star[h]);           // Lemma 10/11
          }
        } else if (!busy) {
          if (same) term = sat_mul(ceil_div64(R + ((gh || literal) ? Jc : 0), Th), s.A[h]);  // L7
        } else {
          if (same) {
            u64 W = s.A[h];                                                        // Lemma 5
            if (gh) W += sat_mul(s.Star[h], nu);                                   // Lemma 4
            term = sat_mul(ceil_div64(R, Th), W);
          }
        }
        part += term;  // each term <= 2^51, at most 8 per lane: no overflow
      }
      const u64 next = base + group_sum<LPT>(part, mask);
      if (next == R) break;
      R = next;
    }
    if (verdict == 0) {
      if (lane == 0) {
        s.R[pos] = R;
        s.prio_out[s.ord[pos] & 0x7fff] = (i64)R;
      }
      __syncwarp(mask);
    } else {
      if (lane == 0) s.prio_out[s.ord[pos] & 0x7fff] = verdict;
      sched = GCAPS_SCHED_NO;
      break;
    }
  }
  __syncwarp(mask);
  if (p.out_wcrt)
    for (int i = lane; i < n; i += LPT) p.out_wcrt[a + i] = s.prio_out[i];
  if (lane == 0) p.out_sched[t] = (uint8_t)sched;
  __syncwarp(mask);
}

// ---------------------------------------------------------------------------------------------
// 32-bit fast path
// ---------------------------------------------------------------------------------------------
// ---- running sums of a segment array, 128 elements per step ------------------------------------
// Lane l takes four consecutive elements (two 16-byte loads), so a warp reads 1 KB contiguous.
// Loads must start on a 16-byte boundary: when the slice starts on an odd element the step begins
// one element early (`par` = 1).  Q[x] receives the sum (modulo 2^32) of elements -par .. x - par;
// Q[-1] is a guard word holding 0.  For 0 <= lo <= hi <= N the sum of elements [lo, hi) is
// Q[hi - 1 + par] - Q[lo - 1 + par]: a borrowed element in front only shifts every entry by the
// same amount, and elements behind the slice only reach entries that are never read.
struct Quad {
  i64 v[4];
};

// Elements e .. e+3 of X, for a slice whose 16-byte pairs all lie inside the array (the common
// case, checked once per taskset by the caller).  Pairs that start at or behind N are not read.
__device__ __forceinline__ void load_quad_inside(const i64 *__restrict__ X, int e, int N, Quad &q) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    longlong2 w = make_longlong2(0, 0);
    if (e + 2 * h < N) w = __ldg(reinterpret_cast<const longlong2 *>(X + e + 2 * h));
    q.v[2 * h] = w.x, q.v[2 * h + 1] = w.y;
  }
}

// The same for a slice at the very edge of its array: only wanted elements inside [lo, hi) are
// touched, everything else reads as 0.
__device__ __noinline__ Quad load_quad_edge(const i64 *__restrict__ X, int e, int N, const i64 *lo,
                                            const i64 *hi) {
  Quad q;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const i64 *ptr = X + e + j;
    q.v[j] = (e + j >= 0 && e + j < N && ptr >= lo && ptr < hi) ? __ldg(ptr) : 0;
  }
  return q;
}

// Narrows a quad to 32 bits, leaves the lane's own running sums in x[0..3] and records in `bad`
// whether a wanted element lies outside [0, 2^26).
__device__ __forceinline__ void narrow_quad(const Quad &q, int e, int N, u32 (&x)[4], u32 &bad) {
  const u32 hi_or = (u32)((u64)q.v[0] >> 32) | (u32)((u64)q.v[1] >> 32) | (u32)((u64)q.v[2] >> 32) |
                    (u32)((u64)q.v[3] >> 32);
  const u32 lo_or = (u32)q.v[0] | (u32)q.v[1] | (u32)q.v[2] | (u32)q.v[3];
  if (hi_or | (lo_or >> 26)) {  // rare: look again, this time only at the elements of this slice
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if ((u32)(e + j) < (u32)N) bad |= (u32)((u64)q.v[j] >> 32) | ((u32)q.v[j] >> 26);
  }
  x[0] = (u32)q.v[0];
  x[1] = x[0] + (u32)q.v[1];
  x[2] = x[1] + (u32)q.v[2];
  x[3] = x[2] + (u32)q.v[3];
}

// True if every 16-byte pair that load_quad_inside would read for this slice is inside the array.
__device__ __forceinline__ bool slice_is_inside(i64 first, int N, int par, i64 total) {
  return (par == 0 || first >= 1) && ((((N + par) & 1) == 0) || first + N < total);
}

// One step (NB blocks of 4*LPT elements) of the running sums of up to two arrays that share their
// offsets, by a group of LPT lanes.  Called by the whole warp (its groups step side by side; a
// group whose slice has ended reads nothing and stores nothing).
template <int LPT, int NB, bool TWO>
__device__ __forceinline__ void prefix_step(const i64 *__restrict__ X0, const i64 *__restrict__ X1,
                                            int e0, int N, int par0, int par1, bool inside,
                                            const i64 *lo0, const i64 *hi0, const i64 *lo1,
                                            const i64 *hi1, u32 *Q0, u32 *Q1, u32 &carry0,
                                            u32 &carry1, u32 &bad, int lane) {
  Quad q0[NB], q1[NB];
  u32 x0[NB][4], x1[NB][4], i0[NB], i1[NB];
  if (inside) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      load_quad_inside(X0, e0 + 4 * LPT * b + 4 * lane - par0, N, q0[b]);
      if (TWO) load_quad_inside(X1, e0 + 4 * LPT * b + 4 * lane - par1, N, q1[b]);
    }
  } else {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      q0[b] = load_quad_edge(X0, e0 + 4 * LPT * b + 4 * lane - par0, N, lo0, hi0);
      if (TWO) q1[b] = load_quad_edge(X1, e0 + 4 * LPT * b + 4 * lane - par1, N, lo1, hi1);
    }
  }
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    narrow_quad(q0[b], e0 + 4 * LPT * b + 4 * lane - par0, N, x0[b], bad);
    i0[b] = x0[b][3];
    if (TWO) {
      narrow_quad(q1[b], e0 + 4 * LPT * b + 4 * lane - par1, N, x1[b], bad);
      i1[b] = x1[b][3];
    }
  }
#pragma unroll
  for (int d = 1; d < LPT; d <<= 1) {  // the scans of all blocks side by side
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const u32 y0 = __shfl_up_sync(kFull, i0[b], d, LPT);
      if (lane >= d) i0[b] += y0;
      if (TWO) {
        const u32 y1 = __shfl_up_sync(kFull, i1[b], d, LPT);
        if (lane >= d) i1[b] += y1;
      }
    }
  }
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const bool wanted = e0 + 4 * LPT * b < N + 1;
    if (LPT == 32 && !wanted) break;  // (the same in every lane)
    const u32 b0 = i0[b] - x0[b][3] + carry0;
    if (wanted)
      *reinterpret_cast<uint4 *>(Q0 + e0 + 4 * LPT * b + 4 * lane) =
          make_uint4(x0[b][0] + b0, x0[b][1] + b0, x0[b][2] + b0, x0[b][3] + b0);
    carry0 += __shfl_sync(kFull, i0[b], LPT - 1, LPT);
    if (TWO) {
      const u32 b1 = i1[b] - x1[b][3] + carry1;
      if (wanted)
        *reinterpret_cast<uint4 *>(Q1 + e0 + 4 * LPT * b + 4 * lane) =
            make_uint4(x1[b][0] + b1, x1[b][1] + b1, x1[b][2] + b1, x1[b][3] + b1);
      carry1 += __shfl_sync(kFull, i1[b], LPT - 1, LPT);
    }
  }
}

// True while the group's slice of N elements has elements at or behind e0 (a warp per taskset), or
// while any group of the warp does.
template <int LPT>
__device__ __forceinline__ bool more_steps(int e0, int N) {
  if constexpr (LPT == 32) return e0 < N;
  return __any_sync(kFull, e0 < N);
}

// An analysis mode known at compile time (converts to int like a run-time mode does).
template <int V>
struct ModeTag {
  __host__ __device__ constexpr operator int() const { return V; }
};

__device__ __forceinline__ void prefetch_l2(const void *ptr) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(ptr));
}

// What a taskset's staging, ordering and aggregation leave in a lane (slot s: position lane + LPT * s);
// info rows (deadline, core) by rank are in shared memory.
template <int SLOTS>
struct TaskValues {
  u32 T[SLOTS], A[SLOTS], Ge[SLOTS], eta[SLOTS];  // period, C+G^m, G^e, GPU segments
  int rank[SLOTS], g0[SLOTS], g1[SLOTS];          // GPU segments of the task within the taskset's slice
  int n, n_gpu, n_rt, n_narrow;  // tasks, GPU-using ones, real-time ones, ranks in single precision
  int Ng, pare;                  // the taskset's G^e slice: elements, odd start
  i64 gfirst;
  bool live;
};

// Stage, order and aggregate, by a group of LPT lanes (8, 16 or a whole warp) per taskset; the whole
// warp calls this and its groups go through every step side by side (`live`: the group has a taskset),
// so that each shuffle, vote and reduction is one instruction for all of them.  False if no group of
// the warp has a taskset that fits the 32-bit path; else o.live says which do.  BC: prefix blocks of
// the CPU segments whose loads are issued together.  ovh_max: the largest epsilon of a GCAPS analysis.
// PREFETCH: the caller has not prefetched the segments; the G^m and G^e slices start their way into L2 as
// soon as their place is known, so that they do not wait for the CPU segments' sums.
// NARROW: a taskset with a period of kNarrowLimit or more is declined before its segments are read.
template <int LPT, int SLOTS, int BC, bool kAnyGcaps, bool PREFETCH = false, bool NARROW = false, class RowsT>
__device__ __forceinline__ bool stage_fast(const KParams &p, bool live, i64 a, int n, u32 *buf, const RowsT rows, int lane,
                                           unsigned int gmask, bool best_effort, u32 ovh_max, TaskValues<SLOTS> &o) {
  typedef FastLayout<LPT, SLOTS> Lay;
  constexpr int MAXN = Lay::MAXN, CAP = Lay::CAP;
  constexpr int BG = 1;
  u32 *Q0 = buf + Lay::kQ0, *Q1 = buf + Lay::kQ1;
  // A group that has no taskset, or declines it, goes on as one with an empty taskset.
#define GCAPS_LEAVE_IF_NONE_LIVE()                                    \
  do {                                                                \
    if (LPT == 32 ? !live : !__any_sync(kFull, live)) return false;   \
    if (!live) n = 0, Nc = 0, Ng = 0;                                 \
  } while (0)

  // ---- stage: per-task scalars, lane = position; rank ----------------------------------------
  u32 (&T)[SLOTS] = o.T, (&A)[SLOTS] = o.A, (&Ge)[SLOTS] = o.Ge, (&eta)[SLOTS] = o.eta;
  int (&rank)[SLOTS] = o.rank, (&g0)[SLOTS] = o.g0, (&g1)[SLOTS] = o.g1, c0[SLOTS], c1[SLOTS];
  int Nc = 0, Ng = 0;
  i64 cfirst, gfirst;
  {
    i64 t64[SLOTS], d64[SLOTS], pr[SLOTS], c64[SLOTS], co[SLOTS], go[SLOTS], cend = 0, gend = 0;
    if (!live) n = 0;
    {
      const i64 k = a + lane;
      const i64 *pT = p.period + k, *pD = p.deadline + k, *pP = p.priority + k, *pK = p.core + k;
      const i64 *pc = p.cseg_off + k, *pg = p.gseg_off + k;
#pragma unroll
      for (int s = 0; s < SLOTS; ++s) {  // all loads of the taskset's per-task arrays in flight
        t64[s] = 2, d64[s] = 1, pr[s] = 0, c64[s] = 0, co[s] = 0, go[s] = 0;
        if (lane + LPT * s < n) {
          t64[s] = pT[LPT * s], d64[s] = pD[LPT * s], pr[s] = pP[LPT * s], c64[s] = pK[LPT * s];
          co[s] = pc[LPT * s], go[s] = pg[LPT * s];
        }
      }
    }
    if (n > 0) cend = p.cseg_off[a + n] - p.cseg_base, gend = p.gseg_off[a + n] - p.gseg_base;
    cfirst = __shfl_sync(kFull, co[0], 0, LPT) - p.cseg_base;
    gfirst = __shfl_sync(kFull, go[0], 0, LPT) - p.gseg_base;
    const i64 Nc64 = cend - cfirst, Ng64 = gend - gfirst;
    if (cfirst < 0 || Nc64 < 0 || cend > p.n_csegs || Nc64 >= CAP || gfirst < 0 || Ng64 < 0 ||
        gend > p.n_gsegs || Ng64 >= CAP)
      live = false;
    Nc = (int)Nc64, Ng = (int)Ng64;
    GCAPS_LEAVE_IF_NONE_LIVE();
    if constexpr (PREFETCH) {
      for (int e = 16 * lane; e < Ng; e += 16 * LPT)
        prefetch_l2(p.gseg_misc + gfirst + e), prefetch_l2(p.gseg_exec + gfirst + e);
    }
    u32 high = 0;  // any set bit: some value does not fit the 32-bit path
    bool ok = true, any_wide = false;
    u32 D[SLOTS], core[SLOTS];
    int prio[SLOTS];
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      const bool v = lane + LPT * s < n;
      const i64 rc = co[s] - p.cseg_base - cfirst, rg = go[s] - p.gseg_base - gfirst;
      const u32 h = (u32)((u64)t64[s] >> 32) | (u32)((u64)d64[s] >> 32) | (u32)((u64)c64[s] >> 32) |
                    (u32)((u64)rc >> 32) | (u32)((u64)rg >> 32) |
                    (u32)(((u64)pr[s] + 0x80000000ull) >> 32);
      T[s] = (u32)t64[s];
      D[s] = (u32)d64[s];
      core[s] = (u32)c64[s];
      prio[s] = v ? (int)pr[s] : (int)0x80000000;
      c0[s] = v ? (int)rc : Nc;
      g0[s] = v ? (int)rg : Ng;
      high |= v ? h : 0u;
      // 2 <= T < 2^26, 1 <= D <= T, core < 2^31, offsets inside the slice
      ok &= !v || (T[s] - 2u < kFastLimit - 2u && D[s] - 1u < T[s] && (int)core[s] >= 0 && (u32)c0[s] <= (u32)Nc &&
                   (u32)g0[s] <= (u32)Ng);
      any_wide |= v && T[s] >= kNarrowLimit;
    }
    // (a wide priority also lands here)
    live = group_all<LPT>(high == 0 && ok && !(NARROW && any_wide), gmask) && live;
    GCAPS_LEAVE_IF_NONE_LIVE();
    if (LPT != 32 && !live) {
#pragma unroll
      for (int s = 0; s < SLOTS; ++s) c0[s] = g0[s] = 0, prio[s] = (int)0x80000000;
    }
    // order: rank by (priority desc, position asc)
    int m = prio[0];
#pragma unroll
    for (int s = 1; s < SLOTS; ++s) m = prio[s] > m ? prio[s] : m;
    int pmax = m;
    if constexpr (LPT == 32) {
      pmax = __reduce_max_sync(kFull, m);
    } else {
#pragma unroll
      for (int d = 1; d < LPT; d <<= 1) {
        const int o = __shfl_xor_sync(kFull, pmax, d);
        pmax = o > pmax ? o : pmax;
      }
    }
    bool dense = true;  // distinct priorities max-n+1 .. max: the rank is max - priority
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      const u32 r = (u32)pmax - (u32)prio[s];
      const bool v = lane + LPT * s < n;
      dense &= !v || r < (u32)n;
      rank[s] = v ? (int)r : MAXN;
    }
    dense = group_all<LPT>(dense, gmask);
    if (dense) {
#pragma unroll
      for (int s = 0; s < SLOTS; ++s)
        if (lane + LPT * s < n) Q0[rank[s]] = (u32)(lane + LPT * s);
    }
    __syncwarp();
    bool uniq = true;
    if (dense) {
#pragma unroll
      for (int s = 0; s < SLOTS; ++s)
        if (lane + LPT * s < n) uniq &= Q0[rank[s]] == (u32)(lane + LPT * s);
    }
    dense = group_all<LPT>(dense && uniq, gmask);
    if (!dense) {  // any priorities: count the tasks that come before
      if constexpr (PREFETCH) {
        // out of shared memory, four at a time: 12,288 tasksets of 80 tasks under GCAPS / RR 149 / 144 -> 64 / 68 us
        // against one after the other out of global memory, which the few warps of a small batch do not hide
        int *const P = reinterpret_cast<int *>(Q0);
        int r[SLOTS];
#pragma unroll
        for (int s = 0; s < SLOTS; ++s) r[s] = 0, P[lane + LPT * s] = prio[s];  // (behind the end: the lowest value)
        __syncwarp();
#pragma unroll 1
        for (int q = 0; q < n; q += 4) {
          const int4 y = *reinterpret_cast<const int4 *>(P + q);
#pragma unroll
          for (int s = 0; s < SLOTS; ++s) {
            const int i = lane + LPT * s;
            r[s] += (y.x > prio[s] || (y.x == prio[s] && q < i)) ? 1 : 0;
            r[s] += (y.y > prio[s] || (y.y == prio[s] && q + 1 < i)) ? 1 : 0;
            r[s] += (y.z > prio[s] || (y.z == prio[s] && q + 2 < i)) ? 1 : 0;
            r[s] += (y.w > prio[s] || (y.w == prio[s] && q + 3 < i)) ? 1 : 0;
          }
        }
#pragma unroll
        for (int s = 0; s < SLOTS; ++s) rank[s] = lane + LPT * s < n ? r[s] : MAXN;
      } else {
#pragma unroll
        for (int s = 0; s < SLOTS; ++s) {
          const int i = lane + LPT * s;
          int r = 0;
#pragma unroll 1
          for (int q = 0; q < n; ++q) {
            const int pq = (int)p.priority[a + q];
            r += (pq > prio[s] || (pq == prio[s] && q < i)) ? 1 : 0;
          }
          rank[s] = i < n ? r : MAXN;
        }
      }
    }
    __syncwarp();
    // best-effort tasks (flag set, priority <= 0) rank behind every real-time task: the ranks
    // from n_rt on are theirs.  n_narrow: the ranks in front of the first period of kNarrowLimit or
    // more.  (Both are kept in spare words in front of Q0's guard entry until the recurrence
    // starts.)
    {
      int n_rt = n;
      if (best_effort) {
#pragma unroll
        for (int s = 0; s < SLOTS; ++s)
          n_rt -= __popc(__ballot_sync(kFull, lane + LPT * s < n && prio[s] <= 0) & gmask);
      }
      int n_narrow = n_rt;
      if (__any_sync(kFull, any_wide)) {
#pragma unroll
        for (int s = 0; s < SLOTS; ++s)
          if (lane + LPT * s < n && T[s] >= kNarrowLimit && rank[s] < n_narrow) n_narrow = rank[s];
#pragma unroll
        for (int d = 1; d < LPT; d <<= 1) {
          const int o = __shfl_xor_sync(kFull, n_narrow, d);
          n_narrow = o < n_narrow ? o : n_narrow;
        }
      }
      if (lane == 0) Q0[-2] = (u32)n_rt, Q0[-3] = (u32)n_narrow;
    }
    // what the row of a rank says about the task itself
#pragma unroll
    for (int s = 0; s < SLOTS; ++s)
      if (lane + LPT * s < n) *reinterpret_cast<uint2 *>(&rows.a(rank[s])) = make_uint2(D[s], core[s]);
  }
  // end offsets: the next task's start (positions beyond n hold the total)
  {
    bool ok = true;
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      const int cn = __shfl_down_sync(kFull, c0[s], 1, LPT), gn = __shfl_down_sync(kFull, g0[s], 1, LPT);
      const int ch = s + 1 < SLOTS ? __shfl_sync(kFull, c0[s + 1 < SLOTS ? s + 1 : s], 0, LPT) : Nc;
      const int gh = s + 1 < SLOTS ? __shfl_sync(kFull, g0[s + 1 < SLOTS ? s + 1 : s], 0, LPT) : Ng;
      c1[s] = lane == LPT - 1 ? ch : cn;
      g1[s] = lane == LPT - 1 ? gh : gn;
      ok &= (u32)(c1[s] - c0[s]) < 64u && (u32)(g1[s] - g0[s]) < 64u;
    }
    live = group_all<LPT>(ok, gmask) && live;
    GCAPS_LEAVE_IF_NONE_LIVE();
  }

  // ---- aggregate ---------------------------------------------------------------------------------
  u32 bad = 0;
  const i64 *__restrict__ Xc = p.cseg_wcet + cfirst;
  const i64 *__restrict__ Xm = p.gseg_misc + gfirst, *__restrict__ Xe = p.gseg_exec + gfirst;
  const int parm = (int)(((uintptr_t)Xm >> 3) & 1), pare = (int)(((uintptr_t)Xe >> 3) & 1);
  if (LPT != 32 && SLOTS == 1 && !live) c0[0] = c1[0] = g0[0] = g1[0] = 0;  // (a group that reads nothing)
  if constexpr ((LPT == 32 && (SLOTS <= 4 || !PREFETCH)) || SLOTS == 1) {
    // A lane adds up the segments of its own tasks, kAtOnce of a kind at a time: independent loads in place of the
    // chain of shuffles of running sums, which a warp per taskset waits for (redundant lines come out of L1).  From
    // the running sums, GCAPS / RR: 1,000 tasksets of 8 tasks 8.2 / 8.4 -> 6.4 / 7.3 us, 12,288 of them 35 / 39 -> 31 /
    // 33, of 80 tasks 51 / 55 -> 47 / 49, of 4 to 192 tasks 97 / 115 -> 73 / 88; GPU priorities of 100,000 tasksets of
    // 80 tasks 720 -> 689; with a plan 100,000 of these 202 / 198 -> 201 / 195.  Four at once from three slots on: 4 to
    // 192 tasks 73 -> 82.  The running sums stay for the one launch over more than 128 tasks, whose registers go from
    // 128 to 168 otherwise (250 tasks under RR 113 -> 130), and for groups of 8 or 16 lanes with two or three slots,
    // whose scans are short (32 tasks under RR 146 -> 149, 30 on one core 96 -> 102).  With one slot, 300,000 tasksets
    // of 2 to 8 tasks: 210 / 217 -> 192 / 198.
    constexpr int kAtOnce = SLOTS <= 2 ? 4 : 2;
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) A[s] = Ge[s] = 0;
#pragma unroll 1
    for (int j0 = 0;; j0 += kAtOnce) {
      bool more = false;
#pragma unroll
      for (int s = 0; s < SLOTS; ++s) more |= c0[s] + j0 < c1[s] || g0[s] + j0 < g1[s];
      if (!__any_sync(kFull, more)) break;
#pragma unroll
      for (int s = 0; s < SLOTS; ++s) {
        i64 w[kAtOnce], m[kAtOnce], e[kAtOnce];
#pragma unroll
        for (int j = 0; j < kAtOnce; ++j) {
          w[j] = m[j] = e[j] = 0;
          if (c0[s] + j0 + j < c1[s]) w[j] = __ldg(Xc + c0[s] + j0 + j);
          if (g0[s] + j0 + j < g1[s]) m[j] = __ldg(Xm + g0[s] + j0 + j), e[j] = __ldg(Xe + g0[s] + j0 + j);
        }
        u32 lo = 0;
#pragma unroll
        for (int j = 0; j < kAtOnce; ++j) {
          bad |= (u32)((u64)w[j] >> 32) | (u32)((u64)m[j] >> 32) | (u32)((u64)e[j] >> 32);
          lo |= (u32)w[j] | (u32)m[j] | (u32)e[j];
          A[s] += (u32)w[j] + (u32)m[j], Ge[s] += (u32)e[j];
        }
        bad |= (lo | A[s] | Ge[s]) >> 26;  // (sums below 2^26 grow by at most eight such values at a time)
      }
    }
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) eta[s] = (u32)(g1[s] - g0[s]);
  } else {
    // running sums of the segment arrays; per-task sums are differences
    const int parc = (int)(((uintptr_t)Xc >> 3) & 1);
    if (lane == 0) Q0[-1] = 0, Q1[-1] = 0;
    {  // CPU segments -> Q0
      const bool inside = slice_is_inside(cfirst, Nc, parc, p.n_csegs);
      u32 carry = 0, unused = 0;
#pragma unroll 1
      for (int e0 = 0; more_steps<LPT>(e0, Nc + parc); e0 += Lay::kStep * BC)
        prefix_step<LPT, BC, false>(Xc, Xc, e0, Nc, parc, parc, inside, p.cseg_wcet, p.cseg_wcet + p.n_csegs,
                               p.cseg_wcet, p.cseg_wcet, Q0, Q0, carry, unused, bad, lane);
    }
    __syncwarp();
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) A[s] = Q0[c1[s] - 1 + parc] - Q0[c0[s] - 1 + parc];
    __syncwarp();
    {  // G^m -> Q0, G^e -> Q1
      const bool inside = slice_is_inside(gfirst, Ng, parm, p.n_gsegs) &&
                          slice_is_inside(gfirst, Ng, pare, p.n_gsegs);
      u32 cm = 0, ce = 0;
#pragma unroll 1
      for (int e0 = 0; more_steps<LPT>(e0, Ng + 1); e0 += Lay::kStep * BG)
        prefix_step<LPT, BG, true>(Xm, Xe, e0, Ng, parm, pare, inside, p.gseg_misc, p.gseg_misc + p.n_gsegs,
                              p.gseg_exec, p.gseg_exec + p.n_gsegs, Q0, Q1, cm, ce, bad, lane);
    }
    __syncwarp();
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      const u32 Gm = Q0[g1[s] - 1 + parm] - Q0[g0[s] - 1 + parm];
      Ge[s] = Q1[g1[s] - 1 + pare] - Q1[g0[s] - 1 + pare];
      eta[s] = (u32)(g1[s] - g0[s]);
      bad |= (A[s] | Gm | Ge[s]) >> 26;
      A[s] += Gm;
      bad |= A[s] >> 26;
    }
  }
  __syncwarp();
  // ---- what does not depend on the timeslice or the overhead ---------------------------------
  int n_gpu = 0;  // N_g
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) n_gpu += __popc(__ballot_sync(kFull, eta[s] > 0) & gmask);
  if (kAnyGcaps) {  // 2 * eps * eta must stay below 2^26 (eta < 64, eps < 2^20: no overflow here)
    #pragma unroll
    for (int s = 0; s < SLOTS; ++s) bad |= (2 * ovh_max * eta[s]) >> 26;
  }
  live = group_all<LPT>(bad == 0, gmask) && live;
  if (LPT == 32 ? !live : !__any_sync(kFull, live)) return false;
  o.live = live, o.n = live ? n : 0, o.n_gpu = n_gpu;
  o.n_rt = live ? (int)Q0[-2] : 0, o.n_narrow = live ? (int)Q0[-3] : 0;
  o.Ng = Ng, o.pare = pare, o.gfirst = gfirst;
#undef GCAPS_LEAVE_IF_NONE_LIVE
  return true;
}

// MODE: 0 GCAPS self-suspension, 1 GCAPS busy-waiting, 2 RR self-suspension, 3 RR busy-waiting.
//
// A group of LPT lanes works on one taskset, side by side with the other groups of its warp.  Until the
// per-task sums are known lane l of a group holds the tasks at positions l, l+LPT, ... ("slots"); then
// every task's values go to the row of its rank in shared memory, where the recurrence finds them.
//
// MASK: bit m set = analysis MODE m is compiled in.  SWEEP: the taskset is staged, ordered and
// aggregated once and then analysed under every (timeslice, overhead) pair q of `sw` and every
// mode m of MASK that sw->enabled names; that analysis writes result block
// q * sw->block_stride + sw->block_of_mode[m] (out_wcrt + block * n_tasks, skipped when out_wcrt
// is null; out_sched + block * n_tasksets).  Without SWEEP, MASK has one bit and the analysis
// takes its constants and outputs from `p`.
//
// Returns, per group, kFastDone (outputs written) or kFastDeclined (some value does not fit the
// 32-bit path or the taskset is invalid; nothing written: the caller runs the exact path).
constexpr int kFastDeclined = 0, kFastDone = 1;
template <int LPT, int SLOTS, int MASK, bool SWEEP = false, bool PREFETCH = false>
__device__ __forceinline__ int analyse_fast(const KParams &p, bool live, i64 t, i64 a, int n, u32 *buf, int lane,
                                            unsigned int gmask, const SweepArgs *sw = nullptr, int q_first = 0,
                                            int q_end = GCAPS_RTA_MAX_SWEEP) {
  typedef FastLayout<LPT, SLOTS> Lay;
  constexpr int MAXN = Lay::MAXN;
  // prefix blocks of the CPU segments whose loads are issued together.  Tasksets of 65..96 tasks
  // with a few GPU segments per task have 200..400 CPU segments: three blocks of 128 cover them
  // in one step where two need a second, mostly empty one (80-task tasksets: -4 % for a GCAPS
  // kernel; the RR kernels, which carry the slice sums too, lose as much to the registers it takes)
  constexpr int BC = SLOTS <= 2 ? SLOTS : ((SLOTS == 3 && (MASK & 12) == 0 && !SWEEP) ? 3 : 2);
  constexpr int BG = 1;
  constexpr bool kAnyGcaps = (MASK & 3) != 0;
  constexpr bool kMulti = (MASK & (MASK - 1)) != 0;
  static_assert(!kMulti || SWEEP, "several analyses per taskset use the sweep loop");
  const bool literal = (p.policy & GCAPS_RTA_LITERAL) != 0;
  const bool best_effort = (p.policy & GCAPS_RTA_BEST_EFFORT) != 0;
  const Rows<LPT, SLOTS, SWEEP> rows{buf};
  u32 *Q0 = buf + Lay::kQ0, *Q1 = buf + Lay::kQ1;
  TaskValues<SLOTS> o;
  if (!stage_fast<LPT, SLOTS, BC, kAnyGcaps, PREFETCH>(p, live, a, n, buf, rows, lane, gmask, best_effort,
                                             SWEEP ? (u32)sw->max_ovh : (u32)p.ovh, o))
    return kFastDeclined;
  live = o.live, n = o.n;
  u32 (&T)[SLOTS] = o.T, (&A)[SLOTS] = o.A, (&Ge)[SLOTS] = o.Ge, (&eta)[SLOTS] = o.eta;
  int (&rank)[SLOTS] = o.rank, (&g0)[SLOTS] = o.g0, (&g1)[SLOTS] = o.g1;
  const int n_gpu = o.n_gpu, Ng = o.Ng, pare = o.pare;
  const i64 gfirst = o.gfirst;
  const i64 *__restrict__ Xe = p.gseg_exec + gfirst;
  const int n_rt = o.n_rt;          // real-time tasks: the ranks that are analysed
  const int n_narrow = o.n_narrow;  // ... of which so many in single precision

  // Eq. 3: running sums of the slices of every pure GPU part for timeslice L (values already
  // checked) into Ps
  auto slice_sums = [&](u32 *Ps, i64 L64, u32 l_mode, u32 l_magic, u32 l_shift) {
    const bool inside = slice_is_inside(gfirst, Ng, pare, p.n_gsegs);
    u32 carry = 0;
    if (lane == 0) Ps[-1] = 0;
#pragma unroll 1
    for (int e0 = 0; more_steps<LPT>(e0, Ng + 1); e0 += Lay::kStep * BG) {
      Quad qe[BG];
      u32 x[BG][4], incl[BG];
#pragma unroll
      for (int b = 0; b < BG; ++b) {
        if (inside) load_quad_inside(Xe, e0 + 4 * LPT * b + 4 * lane - pare, Ng, qe[b]);
        else qe[b] = load_quad_edge(Xe, e0 + 4 * LPT * b + 4 * lane - pare, Ng, p.gseg_exec, p.gseg_exec + p.n_gsegs);
      }
#pragma unroll
      for (int b = 0; b < BG; ++b) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          // a neighbour's element may be large: keep it below 2^26 so the division stays exact
          const u32 w = (u32)qe[b].v[j] & (kFastLimit - 1);
          u32 sq;
          if (l_mode == 0) sq = __umulhi(w + (u32)L64 - 1u, l_magic) >> l_shift;
          else if (l_mode == 1) sq = w;
          else sq = w > 0 ? 1u : 0u;
          x[b][j] = sq + (j > 0 ? x[b][j - 1] : 0u);
        }
        incl[b] = x[b][3];
      }
#pragma unroll
      for (int d = 1; d < LPT; d <<= 1) {
#pragma unroll
        for (int b = 0; b < BG; ++b) {
          const u32 y = __shfl_up_sync(kFull, incl[b], d, LPT);
          if (lane >= d) incl[b] += y;
        }
      }
#pragma unroll
      for (int b = 0; b < BG; ++b) {
        const u32 before = incl[b] - x[b][3] + carry;
        if (e0 + 4 * LPT * b < Ng + 1)
          *reinterpret_cast<uint4 *>(Ps + e0 + 4 * LPT * b + 4 * lane) =
              make_uint4(x[b][0] + before, x[b][1] + before, x[b][2] + before, x[b][3] + before);
        carry += __shfl_sync(kFull, incl[b], LPT - 1, LPT);
      }
    }
    __syncwarp();
  };

  int blocks_made = 0;
  // The recurrence under analysis MODE once the rows are complete, and its outputs, written by
  // position: out_wcrt (unless null in a sweep) and out_sched.
  auto analyse = [&](auto mode_tag, const PairConsts &pc, i64 *out_wcrt, uint8_t *out_sched) {
    constexpr int MODE = mode_tag;  // a ModeTag: every analysis of a kernel gets its own copy
    Outcome out_of = recurrence_narrow<LPT, SLOTS, MODE, SWEEP>(rows, n_narrow, n_gpu, pc, literal, lane, gmask, blocks_made);
    if (out_of.verdict == 0 && n_narrow < n_rt) {
      __syncwarp(gmask);
      out_of = recurrence_wide<LPT, SLOTS, MODE, SWEEP>(buf, n, n_rt, n_narrow, n_gpu, pc, literal, lane, gmask);
    }
    __syncwarp();
    if (!SWEEP || out_wcrt) {
      i64 *const out = out_wcrt + a + lane;
#pragma unroll
      for (int s = 0; s < SLOTS; ++s) {
        if (lane + LPT * s < n) {
          const int r = rank[s];
          i64 value = r >= n_rt ? (i64)GCAPS_WCRT_BEST_EFFORT
                                : (r == out_of.n_done ? (i64)out_of.verdict : (i64)GCAPS_WCRT_SKIPPED);
          if (r < out_of.n_done) value = (i64)rows.R(r);
          out[LPT * s] = value;
        }
      }
    }
    if (live && lane == 0) out_sched[t] = out_of.verdict == 0 ? GCAPS_SCHED_YES : GCAPS_SCHED_NO;
    __syncwarp();
  };

  if constexpr (!SWEEP) {
    // ---- one analysis: constants by position, then everything goes to the rank's rows -----------
    constexpr int MODE = (MASK & 1) ? 0 : (MASK & 2) ? 1 : (MASK & 4) ? 2 : 3;
    constexpr bool kGcaps = MODE < 2;
    PairConsts pc;
    pc.ovh = (u32)p.ovh;  // the fast path needs eps, theta < 2^20
    pc.slot_cost = (u64)p.L + pc.ovh;  // <= 2^41
    u32 sl[SLOTS];               // RR: slices of the task's pure GPU parts (Eq. 3)
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) sl[s] = 0;
    if (!kGcaps) {
      slice_sums(Q0, p.L, p.l_mode, p.l_magic, p.l_shift);
#pragma unroll
      for (int s = 0; s < SLOTS; ++s) sl[s] = Q0[g1[s] - 1 + pare] - Q0[g0[s] - 1 + pare];
      __syncwarp();
    }
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      u32 S, base;
      own_cost<kGcaps>(pc, A[s], Ge[s], eta[s], sl[s], n_gpu, S, base);
      if (lane + LPT * s < n) {
        const u32 flag = eta[s] > 0 ? kRowGpu : 0u;
        rows.b(rank[s]) = make_uint4(T[s], A[s], Ge[s] | flag, S);
        rows.base(rank[s]) = base;
      }
    }
    __syncwarp();
    analyse(ModeTag<MODE>(), pc, p.out_wcrt, p.out_sched);
  } else {
    // ---- several analyses: the tasks go to the rows of their ranks once; S and base of a task are
    // made from the rows when an analysis reaches it (most stop early) ------------------------------
    static_assert(Lay::CAP <= 2048 && Lay::CAP >= 6 * MAXN, "packed segment range, room for the second row");
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      if (lane + LPT * s < n) {
        const u32 flag = eta[s] > 0 ? kRowGpu : 0u;
        rows.b(rank[s]) = make_uint4(T[s], A[s], Ge[s] | flag, 0u);
        // GPU segment range (11 bits each) and number of GPU segments (6 bits), slices
        rows.second(rank[s]) = make_uint2((u32)g0[s] | ((u32)g1[s] << 11) | (eta[s] << 22), 0u);
      }
    }
    __syncwarp();
    i64 sl_L = -1;
    const int enabled = kMulti ? sw->enabled : MASK;
#pragma unroll 1
    for (int q = q_first; q < (q_end < sw->n ? q_end : sw->n); ++q) {
      const i64 L64 = sw->q[q].L;
      PairConsts pc;
      pc.ovh = (u32)sw->q[q].ovh;  // the fast path needs eps, theta < 2^20
      pc.slot_cost = (u64)L64 + pc.ovh;
      auto analyse_as = [&](auto mode_tag) {
        constexpr int MODE = mode_tag;
        constexpr bool kGcaps = MODE < 2;
        const int block = q * sw->block_stride + sw->block_of_mode[MODE];
        i64 *const out_wcrt = p.out_wcrt ? p.out_wcrt + (i64)block * p.n_tasks : nullptr;
        uint8_t *const out_sched = p.out_sched + (i64)block * p.n_tasksets;
        if (!kGcaps && L64 != sl_L) {
          sl_L = L64;
          slice_sums(Q1, L64, sw->q[q].l_mode, sw->q[q].l_magic, sw->q[q].l_shift);
#pragma unroll
          for (int s = 0; s < SLOTS; ++s) {
            const int r = lane + LPT * s;
            if (r < n) {
              const u32 g = rows.second(r).x;
              rows.second(r).y = Q1[(int)((g >> 11) & 0x7ffu) - 1 + pare] - Q1[(int)(g & 0x7ffu) - 1 + pare];
            }
          }
          __syncwarp();
        }
        analyse(mode_tag, pc, out_wcrt, out_sched);
      };
      if ((MASK & 1) && (enabled & 1)) analyse_as(ModeTag<0>());
      if ((MASK & 2) && (enabled & 2)) analyse_as(ModeTag<1>());
      if ((MASK & 4) && (enabled & 4)) analyse_as(ModeTag<2>());
      if ((MASK & 8) && (enabled & 8)) analyse_as(ModeTag<3>());
    }
  }
  return live ? kFastDone : kFastDeclined;
}

// What a warp knows in advance about one taskset of a chunk (kept in shared memory).
struct Ahead {
  i64 a;           // first task
  i64 c_lo, g_lo;  // first CPU segment, first GPU segment
  u32 t;           // taskset index
  u32 packed;      // tasks (bits 0-8) | CPU segments (9-19) | GPU segments (20-30) | offsets in range (31)
};
static_assert(sizeof(Ahead) == 32, "two 16-byte rows");
constexpr int kMaxAhead = 16;  // tasksets of one pull
constexpr int kAheadWords = 2 * kMaxAhead * (int)(sizeof(Ahead) / sizeof(u32));  // two chunks

constexpr u32 kNoTaskset = 0xffffffffu;

// Looks up one taskset (or none) of a bin for at most MAXN tasks and CAP-1 segments of a kind.  One whose
// first or last offset lies outside its array has bit 31 of `packed` clear, and the exact path says what it
// is: the stages see differences of offsets only, and without a segment all of those are 0.
template <int MAXN, int CAP>
__device__ __forceinline__ Ahead look_up_taskset(const KParams &p, u32 t) {
  static_assert(MAXN <= 256 && CAP <= 2048, "fields of Ahead::packed");
  Ahead me;
  me.a = 0, me.c_lo = me.g_lo = 0, me.t = t, me.packed = 0;
  if (t != kNoTaskset) {
    me.a = p.task_off[t] - p.task_base;
    const i64 b = p.task_off[(i64)t + 1] - p.task_base;
    if (me.a >= 0 && b > me.a && b <= p.n_tasks && b - me.a <= MAXN) {
      me.c_lo = p.cseg_off[me.a] - p.cseg_base, me.g_lo = p.gseg_off[me.a] - p.gseg_base;
      const i64 c_hi = p.cseg_off[b] - p.cseg_base, g_hi = p.gseg_off[b] - p.gseg_base;
      const bool in_range = me.c_lo >= 0 && c_hi >= me.c_lo && c_hi <= p.n_csegs && me.g_lo >= 0 && g_hi >= me.g_lo &&
                            g_hi <= p.n_gsegs;
      // (too many segments for the 32-bit path: none are fetched in advance)
      const u32 nc = in_range && c_hi - me.c_lo < CAP ? (u32)(c_hi - me.c_lo) : 0u;
      const u32 ng = in_range && g_hi - me.g_lo < CAP ? (u32)(g_hi - me.g_lo) : 0u;
      me.packed = (u32)(b - me.a) | (nc << 9) | (ng << 20) | (in_range ? 0x80000000u : 0u);
    }
  }
  return me;
}

// The segment slices start their way into L2 (16 elements per line, only addresses inside the
// arrays); the per-task loads follow at once, so that the running sums later wait for L2 rather
// than for DRAM.
template <int LPT>
__device__ __forceinline__ void prefetch_segments(const KParams &p, const Ahead &me, int lane) {
  const int nc = (int)((me.packed >> 9) & 0x7ffu), ng = (int)((me.packed >> 20) & 0x7ffu);
  for (int e = 16 * lane; e < nc; e += 16 * LPT) prefetch_l2(p.cseg_wcet + me.c_lo + e);
  for (int e = 16 * lane; e < ng; e += 16 * LPT)
    prefetch_l2(p.gseg_misc + me.g_lo + e), prefetch_l2(p.gseg_exec + me.g_lo + e);
}

// blocks per SM the register allocation aims at: more warps in flight matter more here than a
// few spilled values, because every phase is a chain of dependent instructions and the loads of
// a taskset can only be hidden behind the work of other warps
__host__ __device__ constexpr int min_blocks(int slots) {
  return slots <= 3 ? 6 : slots == 4 ? 4 : slots == 6 ? 3 : 2;
}

// The exact path once per (timeslice, overhead) pair q_first .. q_end-1 and analysis of a sweep.
template <int LPT, int MAXN, int MASK>
__device__ __forceinline__ void exact_by_pair(const KParams &p, const SweepArgs &sw, i64 t, GroupSmem<MAXN> &s, int lane,
                                              unsigned int gmask, int q_first, int q_end) {
  constexpr bool kMulti = (MASK & (MASK - 1)) != 0;
  const int enabled = kMulti ? sw.enabled : MASK;
#pragma unroll 1
  for (int q = q_first; q < q_end; ++q) {
#pragma unroll 1
    for (int m = 0; m < 4; ++m) {
      if (!((MASK & enabled) >> m & 1)) continue;
      const int block = q * sw.block_stride + sw.block_of_mode[m];
      KParams pq = p;
      pq.policy = (p.policy & ~(0xff | GCAPS_RTA_BUSY)) | (m >= 2 ? GCAPS_POLICY_RR : GCAPS_POLICY_GCAPS) |
                  ((m & 1) ? GCAPS_RTA_BUSY : 0);
      pq.L = sw.q[q].L, pq.ovh = sw.q[q].ovh;
      pq.out_wcrt = p.out_wcrt ? p.out_wcrt + (i64)block * p.n_tasks : nullptr;
      pq.out_sched = p.out_sched + (i64)block * p.n_tasksets;
      analyse_taskset<LPT, MAXN>(pq, t, s, lane, gmask);
      __syncwarp(gmask);
    }
  }
}

// One size bin, worked through by all warps of a persistent launch.  A warp is 32/LPT groups of
// LPT lanes; every group analyses one taskset at a time.  Warps pull chunks of taskset indices
// from the bin's counter; the index, task range and first segment offsets of the next chunk are
// fetched while the current one is analysed.
template <int LPT, int SLOTS, int MASK, bool SWEEP = false>
__device__ __forceinline__ void run_bin(const KParams &p, int bin, u32 *warp_buf, Ahead *ahead,
                                        const SweepArgs *sw = nullptr) {
  typedef FastLayout<LPT, SLOTS> Lay;
  constexpr int MAXN = LPT * SLOTS;
  constexpr int G = 32 / LPT;  // groups per warp
  static_assert(sizeof(GroupSmem<MAXN>) <= sizeof(u32) * Lay::kWords, "exact path fits");
  const int lane32 = threadIdx.x & 31, group = lane32 / LPT, lane = lane32 % LPT;
  const unsigned int gmask = LPT == 32 ? kFull : (((1u << LPT) - 1u) << (group * LPT));
  u32 *buf = warp_buf + group * Lay::kWords;
  // (the last bin ends with the permutation, also where tiles list their left-over tasksets in it from the end on)
  const unsigned int count = p.hdr->bin_count[bin], start = bin == kRestLarge ? (unsigned int)p.n_tasksets - count : p.hdr->bin_start[bin];
  if (count == 0) return;
  // keeps 2*eps*eta and (eta+1)*eps in 32 bits
  const bool fast_call = (SWEEP ? sw->max_ovh : p.ovh) < (1 << 20);
  // tasksets per pull: up to 8 per group when the bin is large, fewer when that would leave warps
  // without work
  const unsigned int n_groups = gridDim.x * (kBlockThreads / 32) * G;
  const int rounds = count >= 32 * n_groups ? (G == 1 ? 8 : kMaxAhead / G)
                                      : (count >= 8 * n_groups ? 4 / (G > 2 ? 2 : 1) : 1);
  const int chunk = rounds * G;  // <= kMaxAhead

  // lanes 0..chunk-1 each look up one taskset of a chunk and leave what they found in `slot`
  auto look_up = [&](unsigned int first, Ahead *slot) {
    if (lane32 < chunk) {
      u32 t = kNoTaskset;
      if (first < count && first + lane32 < count) t = p.perm[start + first + lane32];
      slot[lane32] = look_up_taskset<MAXN, Lay::CAP>(p, t);
    }
    __syncwarp();
  };

  unsigned int first = 0;
  if (lane32 == 0) first = atomicAdd(&p.hdr->next[bin], (unsigned int)chunk);
  first = __shfl_sync(kFull, first, 0);
  int which = 0;
  look_up(first, ahead);
#pragma unroll 1
  while (first < count) {
    unsigned int nfirst = 0;
    if (lane32 == 0) nfirst = atomicAdd(&p.hdr->next[bin], (unsigned int)chunk);
    const Ahead *cur = ahead + which * kMaxAhead;
    Ahead *nxt = ahead + (which ^ 1) * kMaxAhead;
    const int in_chunk = count - first < (unsigned int)chunk ? (int)(count - first) : chunk;
    const int in_rounds = (in_chunk + G - 1) / G;
#pragma unroll 1
    for (int c = 0; c < in_rounds; ++c) {
      if (c == 1 || in_rounds == 1) {  // the next chunk's index has arrived by now
        nfirst = __shfl_sync(kFull, nfirst, 0);
        look_up(nfirst, nxt);
      }
      const int mine = c * G + group;
      const Ahead me = cur[mine < in_chunk ? mine : 0];
      const bool have = mine < in_chunk;
      const i64 t = (i64)me.t;
      const int n = (int)(me.packed & 0x1ffu);
      const bool fast = have && fast_call && (me.packed >> 31) != 0;
      if (have) prefetch_segments<LPT>(p, me, lane);
      int how = kFastDeclined;
      if (fast_call) how = analyse_fast<LPT, SLOTS, MASK, SWEEP>(p, fast, t, me.a, n, buf, lane, gmask, sw);
      __syncwarp();
      if (have && how != kFastDone) {
        if (!SWEEP) {
          // the exact path reads task_off again and validates everything itself
          analyse_taskset<LPT, MAXN>(p, t, *reinterpret_cast<GroupSmem<MAXN> *>(buf), lane, gmask);
        } else {
          exact_by_pair<LPT, MAXN, MASK>(p, *sw, t, *reinterpret_cast<GroupSmem<MAXN> *>(buf), lane, gmask, 0, sw->n);
        }
      }
      __syncwarp();
    }
    first = nfirst;
    which ^= 1;
  }
}

// shared memory of one warp for the bins a kernel covers
template <int LPT, int SLOTS>
__host__ __device__ constexpr int bin_warp_words() {
  return (32 / LPT) * FastLayout<LPT, SLOTS>::kWords;
}
__host__ __device__ constexpr int cmax(int a, int b) { return a > b ? a : b; }
constexpr int kSmallWarpWords =
    cmax(cmax(bin_warp_words<8, 1>(), bin_warp_words<8, 2>()),
         cmax(bin_warp_words<8, 3>(), bin_warp_words<16, 2>())) + kAheadWords;

// ---- behind tiles: the tasksets that these listed as left over, or all size bins where the batch was none for tiles ----------
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
#endif  // GCAPS_RTA_DEVICE_CUH_
