// gcaps_gpu_priority.cu -- the GCAPS analysis with a separate priority for GPU segments, and the
// Audsley-style search for those priorities (GCAPS, ECRTS 2024, arXiv 2406.05221, Sec. 5.3 and
// Sec. 6.4), for NVIDIA B200 (sm_100a).
//
// Sec. 6.4 replaces R_h by D_h in every jitter, so each pair (J, W) of an interferer is a
// constant of the taskset and the tasks of a taskset can be bounded in any order.  A group of 8,
// 16 or 32 lanes works on one taskset (tasksets are binned by size with the same plan as the
// default analysis); lane l of the group keeps, in registers, what its tasks (positions l,
// l + lanes, ...) contribute as interferers: 1/T_h, the same-core pairs (J^c_h, C_h + G^{m*}_h) and
// (J^g_h, G^e_h), and the other-core pair (J^g_h, G^{e*}_h).  Bounding one task is then: a per-lane
// choice of which pairs apply (same core and higher CPU priority; or "still without a level"), and
// sweeps summed across the group.
//
// search_narrow does the search for tasksets whose periods all lie below kNarrowLimit: staged and
// aggregated like the default analysis (stage_fast), bounded in packed single precision with exact
// integer results (see rta_recurrence.cuh).  All others, and given priorities, go through integers
// (analyse_gpu_priority): 32-bit while all values of a taskset are below 2^26 us, else the same loop in
// saturating 64-bit.  The kernels of the size bins hold only the one or the other: out of line in the
// search's kernels, with their registers and shared memory, the integer code took up to 2.7 times as long.
#include <cuda_runtime.h>
#include <stdint.h>

#include "rta_device.cuh"

using namespace gcaps_detail;

namespace {

struct GpParams {
  KParams k;
  const i64 *gpu_prio_in;
  i64 *gpu_prio_out;
};

// Per-taskset shared memory of a group, by position.
template <int MAXN>
struct GpSmem {
  i64 key[MAXN];   // priorities while ranking
  i64 base[MAXN];  // C_i + G*_i + B^C_i
  i64 D[MAXN];
  int core[MAXN];
  short cpu_rank[MAXN];     // 0 = highest CPU priority, ties by position
  short gpu_rank[MAXN];     // the same for the given GPU priorities
  short by_cpu_rank[MAXN];  // CPU rank -> position
  unsigned char uses_gpu[MAXN];
  // search: bit r set = the task of CPU rank r has no level yet and no task of lower CPU priority
  // on its core is without one, i.e. it may take the next level (the same-core rule of Sec. 5.3)
  unsigned int cand[8];
};

// Largest r < below with bit r set in the 256-bit set `bits`, or -1.
__device__ __forceinline__ int highest_below(const unsigned int *bits, int below) {
  for (int w = (below - 1) >> 5; w >= 0; --w) {
    unsigned int m = bits[w];
    if (w == (below - 1) >> 5) m &= (2u << ((below - 1) & 31)) - 1u;  // (2u << 31 wraps to 0: all ones)
    if (m) return 32 * w + 31 - __clz((int)m);
  }
  return -1;
}

// What a lane knows about its S tasks as interferers (slot s: position lane + LPT * s).
template <int S>
struct GpLane {
  u64 T[S];
  u64 Kc[S], Kg[S];          // J^c_h + T_h - 1, J^g_h + T_h - 1 (the ceiling folded in)
  u64 Wc[S], We[S], Wes[S];  // C_h + G^m_h (+ 2 eps eta_h unless busy-waiting), G^e_h, G^{e*}_h
  u32 magic[S], shift[S];    // reciprocal of T_h (32-bit path)
  int core[S], cpu_rank[S];
  bool gpu[S], valid[S];
};

template <int LPT>
__device__ __forceinline__ u32 sum32(u32 v, unsigned int gmask) {
  if constexpr (LPT == 32) {
    return __reduce_add_sync(gmask, v);
  } else {
#pragma unroll
    for (int d = LPT / 2; d >= 1; d >>= 1) v += __shfl_xor_sync(gmask, v, d, LPT);
    return v;
  }
}

// Bound of task i (core_i, CPU rank rank_i, GPU-using gi, constant part `base`, deadline Di) when
// the tasks flagged in above[] have a higher GPU-segment priority: the recurrence of Sec. 6.3
// with hp() by GPU priority and D_h in the jitters (Sec. 6.4).  Returns the bound,
// GCAPS_WCRT_MISS or GCAPS_WCRT_ITER_LIMIT, the same value in every lane of the group.
template <int LPT, int S, bool FAST>
__device__ __forceinline__ i64 bound_of(const GpLane<S> &me, int lane, unsigned int gmask, int i,
                                        int core_i, int rank_i, bool gi, u64 base, u64 Di,
                                        const bool (&above)[S], bool busy, bool literal) {
  // the (J, W) pairs of this lane's tasks; W = 0 where a pair does not apply
  u64 Ka[S], Wa[S], Wb[S];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const int h = lane + LPT * s;
    const bool hpp = me.valid[s] && h != i && me.core[s] == core_i && me.cpu_rank[s] < rank_i;
    const bool hpg = me.valid[s] && h != i && above[s] && !hpp;  // hp(tau_i) of Sec. 6.4 minus hpp
    Ka[s] = me.Kc[s], Wa[s] = 0, Wb[s] = 0;
    if (!busy) {
      if (hpp) Wa[s] = me.Wc[s];                      // Lemma 15 (jitter 0 for a CPU-only tau_h)
      if (hpp && me.gpu[s] && gi) Wb[s] = me.We[s];   // Lemma 13, same core
      if (hpg && me.gpu[s] && gi) Wb[s] = me.Wes[s];  // Lemma 13, other cores
    } else {
      if (hpp) {
        Ka[s] = me.T[s] - 1;                                                       // no jitter
        Wa[s] = me.Wc[s] + ((me.gpu[s] && (gi || !literal)) ? me.Wes[s] : 0);      // Lemmas 12, 10
      } else if (hpg && me.gpu[s]) {
        Wb[s] = me.Wes[s];                                                         // Lemmas 10, 11
      }
    }
  }
  u64 R = base;
  i64 sweeps = 0;
  for (;;) {
    if (R > Di) return GCAPS_WCRT_MISS;
    if (sweeps >= GCAPS_RTA_ITER_CAP) return GCAPS_WCRT_ITER_LIMIT;
    sweeps += 1;
    u64 next;
    if (FAST) {  // R <= D_i < 2^26, K < 2^27: the dividend stays below 2^28
      u64 acc = 0;
#pragma unroll
      for (int s = 0; s < S; ++s) {
        acc += (u64)(__umulhi((u32)R + (u32)Ka[s], me.magic[s]) >> me.shift[s]) * (u32)Wa[s];
        acc += (u64)(__umulhi((u32)R + (u32)me.Kg[s], me.magic[s]) >> me.shift[s]) * (u32)Wb[s];
      }
      const u32 part = acc > (u64)kFastClamp ? kFastClamp : (u32)acc;
      next = base + sum32<LPT>(part, gmask);
    } else {
      u64 part = 0;
#pragma unroll
      for (int s = 0; s < S; ++s) {
        if (Wa[s]) part += sat_mul((R + Ka[s]) / me.T[s], Wa[s]);
        if (Wb[s]) part += sat_mul((R + me.Kg[s]) / me.T[s], Wb[s]);
      }
      next = base + group_sum<LPT>(part > kClamp ? kClamp : part, gmask);
    }
    if (next == R) return (i64)R;
    R = next;
  }
}

// What the lane's tasks contribute, and what the group looks up by position, from the tasks' values.
template <int LPT, int S>
__device__ __forceinline__ void lane_values(u64 eps, bool busy, bool fits32, const u64 (&T)[S], const u64 (&D)[S],
                                            const u64 (&A)[S], const u64 (&Ge)[S], const u64 (&Star)[S], const int (&eta)[S],
                                            const int (&core)[S], const bool (&valid)[S], GpLane<S> &me,
                                            GpSmem<LPT * S> &sm, int lane) {
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const int i = lane + LPT * s;
    const bool gh = eta[s] > 0;
    // Sec. 6.4: J^c_h = D_h - (C_h + G^m_h), J^g_h = D_h - G^e_h (a task whose own execution
    // exceeds its deadline has no such slack: 0); a CPU-only tau_h has no J^c (Lemma 15)
    const u64 Jc = (gh && D[s] > A[s]) ? D[s] - A[s] : 0, Jg = D[s] > Ge[s] ? D[s] - Ge[s] : 0;
    me.T[s] = T[s], me.Kc[s] = Jc + T[s] - 1, me.Kg[s] = Jg + T[s] - 1;
    me.Wc[s] = A[s] + ((gh && !busy) ? Star[s] : 0);  // Lemma 15: C_h + G^{m*}_h; Lemma 12: C_h + G^m_h
    me.We[s] = Ge[s], me.Wes[s] = Ge[s] + Star[s];
    me.core[s] = core[s], me.gpu[s] = gh, me.valid[s] = valid[s];
    me.magic[s] = 0, me.shift[s] = 0;
    if (fits32) make_reciprocal((u32)T[s], me.magic[s], me.shift[s]);
    if (valid[s]) {
      sm.cpu_rank[i] = (short)me.cpu_rank[s];
      sm.by_cpu_rank[me.cpu_rank[s]] = (short)i;
      sm.uses_gpu[i] = gh ? 1 : 0;
      sm.base[i] = (i64)(A[s] + Ge[s] + Star[s] + ((u64)eta[s] + 1) * eps);  // C_i + G*_i + B^C_i
      sm.D[i] = (i64)D[s];
    }
  }
}

// The bound of the task at position i by bound_of, in 32 bits where its values fit.
template <int LPT, int S>
__device__ __forceinline__ i64 bound_at(const GpLane<S> &me, const GpSmem<LPT * S> &sm, int i, const bool (&above)[S],
                                        bool fits32, bool busy, bool literal, int lane, unsigned int gmask) {
  const int core_i = sm.core[i], rank_i = sm.cpu_rank[i];
  const bool gi = sm.uses_gpu[i] != 0;
  const u64 bi = (u64)sm.base[i], Di = (u64)sm.D[i];
  if (fits32 && bi < kFastClamp)
    return bound_of<LPT, S, true>(me, lane, gmask, i, core_i, rank_i, gi, bi, Di, above, busy, literal);
  return bound_of<LPT, S, false>(me, lane, gmask, i, core_i, rank_i, gi, bi, Di, above, busy, literal);
}

// The search of Sec. 5.3 in integers: levels from the lowest.  Returns GCAPS_SCHED_YES or _NO.
template <int LPT, int S>
__device__ __forceinline__ int search_levels(const GpParams &g, i64 a, int n, const GpLane<S> &me, const int (&core)[S],
                                             const bool (&valid)[S], GpSmem<LPT * S> &sm, bool fits32, bool busy, bool literal,
                                             int lane, unsigned int gmask) {
  const KParams &p = g.k;
  int sched = GCAPS_SCHED_YES;
  bool unplaced[S];
  if (lane < 8) sm.cand[lane] = 0;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    unplaced[s] = valid[s];
    if (valid[s]) {
      p.out_wcrt[a + lane + LPT * s] = GCAPS_WCRT_MISS;
      g.gpu_prio_out[a + lane + LPT * s] = 0;
    }
  }
  __syncwarp(gmask);
  {  // the lowest CPU priority of every core starts as a candidate
    bool lowest[S];
#pragma unroll
    for (int s = 0; s < S; ++s) lowest[s] = valid[s];
    for (int q = 0; q < n; ++q) {
      const int core_q = sm.core[q], rank_q = sm.cpu_rank[q];
#pragma unroll
      for (int s = 0; s < S; ++s) lowest[s] &= !(core_q == core[s] && rank_q > me.cpu_rank[s]);
    }
#pragma unroll
    for (int s = 0; s < S; ++s)
      if (lowest[s]) atomicOr(&sm.cand[me.cpu_rank[s] >> 5], 1u << (me.cpu_rank[s] & 31));
  }
  __syncwarp(gmask);
  for (int level = 1; level <= n && sched == GCAPS_SCHED_YES; ++level) {
    bool placed = false;
    int want = n;
    while (!placed) {  // candidates from the lowest CPU priority upwards
      want = highest_below(sm.cand, want);
      if (want < 0) break;
      const int c = sm.by_cpu_rank[want];
      // every other unplaced task above c (c itself is skipped)
      const i64 r = bound_at<LPT, S>(me, sm, c, unplaced, fits32, busy, literal, lane, gmask);
      if (r >= 0) {
        placed = true;
        const int core_c = sm.core[c];
        int next = -1;  // the task of c's core that becomes a candidate now
#pragma unroll
        for (int s = 0; s < S; ++s) {
          if (lane + LPT * s == c) {
            unplaced[s] = false;
            p.out_wcrt[a + c] = r;
            g.gpu_prio_out[a + c] = (i64)level;
          }
          if (unplaced[s] && core[s] == core_c && me.cpu_rank[s] < want && me.cpu_rank[s] > next)
            next = me.cpu_rank[s];
        }
#pragma unroll
        for (int d = LPT / 2; d >= 1; d >>= 1) {
          const int other = __shfl_xor_sync(gmask, next, d, LPT);
          next = other > next ? other : next;
        }
        __syncwarp(gmask);
        if (lane == 0) {
          sm.cand[want >> 5] &= ~(1u << (want & 31));
          if (next >= 0) sm.cand[next >> 5] |= 1u << (next & 31);
        }
        __syncwarp(gmask);
      }
    }
    if (!placed) sched = GCAPS_SCHED_NO;
  }
  return sched;
}

// One taskset in integers from global memory, by a group of LPT lanes.  ASSIGN: the search, else the given
// GPU priorities.
template <int LPT, int S, bool ASSIGN>
__device__ __forceinline__ void analyse_gpu_priority(const GpParams &g, i64 t, GpSmem<LPT * S> &sm, int lane,
                                                     unsigned int gmask) {
  constexpr int MAXN = LPT * S;
  const KParams &p = g.k;
  const bool busy = (p.policy & GCAPS_RTA_BUSY) != 0, literal = (p.policy & GCAPS_RTA_LITERAL) != 0;
  const u64 eps = (u64)p.ovh;
  const i64 a = p.task_off[t], b = p.task_off[t + 1];
  if (a < 0 || b < a || b > p.n_tasks || b - a > MAXN) {
    // (a taskset of more than MAXN tasks can only reach the largest bin, where MAXN is the limit)
    if (lane == 0) p.out_sched[t] = GCAPS_SCHED_INVALID;
    return;
  }
  const int n = (int)(b - a);

  // ---- stage, validate, aggregate (task model of Sec. 4) ------------------------------------
  int bad = 0;
  bool fits32 = eps < (1u << 20);
  u64 T[S], D[S], A[S], Ge[S], Star[S];
  int eta[S], core[S];
  bool valid[S];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const int i = lane + LPT * s;
    valid[s] = i < n;
    T[s] = 2, D[s] = 1, A[s] = 0, Ge[s] = 0, Star[s] = 0, eta[s] = 0, core[s] = -1;
    if (valid[s]) {
      const i64 k = a + i;
      const i64 Ti = p.period[k], Di = p.deadline[k], c = p.core[k];
      if (Ti < 1 || Ti > GCAPS_RTA_MAX_TIME) bad |= GCAPS_BAD_PERIOD;
      if (Di < 1 || Di > Ti) bad |= GCAPS_BAD_DEADLINE;
      if (c < 0 || c > GCAPS_RTA_MAX_CORE) bad |= GCAPS_BAD_CORE;
      const i64 c0 = p.cseg_off[k], c1 = p.cseg_off[k + 1], g0 = p.gseg_off[k], g1 = p.gseg_off[k + 1];
      const bool seg_ok = !(c0 < 0 || c1 < c0 || c1 > p.n_csegs || c1 - c0 > GCAPS_RTA_MAX_SEGMENTS ||
                            g0 < 0 || g1 < g0 || g1 > p.n_gsegs || g1 - g0 > GCAPS_RTA_MAX_SEGMENTS);
      u64 C = 0, Gm = 0, Gx = 0;
      if (seg_ok) {
#pragma unroll 4
        for (i64 j = c0; j < c1; ++j) {
          const i64 w = p.cseg_wcet[j];
          if (w < 0 || w > GCAPS_RTA_MAX_TIME) bad |= GCAPS_BAD_WCET;
          C += (u64)w;
        }
#pragma unroll 4
        for (i64 j = g0; j < g1; ++j) {
          const i64 m = p.gseg_misc[j], e = p.gseg_exec[j];
          if (m < 0 || m > GCAPS_RTA_MAX_TIME || e < 0 || e > GCAPS_RTA_MAX_TIME) bad |= GCAPS_BAD_WCET;
          Gm += (u64)m, Gx += (u64)e;
        }
      } else {
        bad |= GCAPS_BAD_SEG_RANGE;
      }
      eta[s] = seg_ok ? (int)(g1 - g0) : 0;
      T[s] = (u64)Ti, D[s] = (u64)Di, A[s] = C + Gm, Ge[s] = Gx, core[s] = (int)c;
      Star[s] = 2 * eps * (u64)eta[s];
      sm.key[i] = p.priority[k];
      sm.core[i] = (int)c;
      fits32 = fits32 && Ti >= 2 && Ti < (i64)kFastLimit && eta[s] < 64 && A[s] + Star[s] < kFastLimit &&
               Gx + Star[s] < kFastLimit;
    }
  }
  bad = group_or<LPT>(bad, gmask);
  fits32 = __all_sync(gmask, fits32);
  __syncwarp(gmask);
  if (bad) {
#pragma unroll
    for (int s = 0; s < S; ++s)
      if (valid[s]) {
        p.out_wcrt[a + lane + LPT * s] = GCAPS_WCRT_INVALID;
        if (g.gpu_prio_out) g.gpu_prio_out[a + lane + LPT * s] = 0;
      }
    if (lane == 0) p.out_sched[t] = GCAPS_SCHED_INVALID;
    return;
  }
  // ---- CPU ranks: larger priority first, ties by position -----------------------------------
  GpLane<S> me;
  // distinct priorities hi-n+1 .. hi (what a numbering by period gives): the rank is hi - priority
  i64 hi = INT64_MIN;
#pragma unroll
  for (int s = 0; s < S; ++s)
    if (valid[s] && sm.key[lane + LPT * s] > hi) hi = sm.key[lane + LPT * s];
#pragma unroll
  for (int d = LPT / 2; d >= 1; d >>= 1) {
    const i64 other = __shfl_xor_sync(gmask, hi, d, LPT);
    hi = other > hi ? other : hi;
  }
  bool dense = true;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const u64 r = valid[s] ? (u64)hi - (u64)sm.key[lane + LPT * s] : 0;
    dense &= r < (u64)n;
    me.cpu_rank[s] = (int)(r < (u64)n ? r : 0);
  }
  dense = __all_sync(gmask, dense);
  if (dense) {  // ... and no rank taken twice
#pragma unroll
    for (int s = 0; s < S; ++s)
      if (valid[s]) sm.by_cpu_rank[me.cpu_rank[s]] = (short)(lane + LPT * s);
    __syncwarp(gmask);
    bool uniq = true;
#pragma unroll
    for (int s = 0; s < S; ++s)
      if (valid[s]) uniq &= sm.by_cpu_rank[me.cpu_rank[s]] == (short)(lane + LPT * s);
    dense = __all_sync(gmask, uniq);
    __syncwarp(gmask);
  }
  if (!dense) {  // any priorities: count the tasks that come before
    i64 mine[S];
#pragma unroll
    for (int s = 0; s < S; ++s) mine[s] = valid[s] ? sm.key[lane + LPT * s] : 0, me.cpu_rank[s] = 0;
    for (int q = 0; q < n; ++q) {
      const i64 kq = sm.key[q];
#pragma unroll
      for (int s = 0; s < S; ++s)
        me.cpu_rank[s] += (valid[s] && (kq > mine[s] || (kq == mine[s] && q < lane + LPT * s))) ? 1 : 0;
    }
  }
  __syncwarp(gmask);
  lane_values<LPT, S>(eps, busy, fits32, T, D, A, Ge, Star, eta, core, valid, me, sm, lane);
  __syncwarp(gmask);
  int sched = GCAPS_SCHED_YES;
  if constexpr (!ASSIGN) {
    // ---- the given GPU priorities ---------------------------------------------------------------
#pragma unroll
    for (int s = 0; s < S; ++s)
      if (valid[s]) sm.key[lane + LPT * s] = g.gpu_prio_in[a + lane + LPT * s];
    __syncwarp(gmask);
    int gpu_rank[S];
    {
      i64 mine[S];
#pragma unroll
      for (int s = 0; s < S; ++s) mine[s] = valid[s] ? sm.key[lane + LPT * s] : 0, gpu_rank[s] = 0;
      for (int q = 0; q < n; ++q) {
        const i64 kq = sm.key[q];
#pragma unroll
        for (int s = 0; s < S; ++s)
          gpu_rank[s] += (valid[s] && (kq > mine[s] || (kq == mine[s] && q < lane + LPT * s))) ? 1 : 0;
      }
#pragma unroll
      for (int s = 0; s < S; ++s)
        if (valid[s]) sm.gpu_rank[lane + LPT * s] = (short)gpu_rank[s];
    }
    __syncwarp(gmask);
    int broken = 0;  // same core: the GPU order must equal the CPU order (Sec. 5.3)
    for (int q = 0; q < n; ++q) {
      const int core_q = sm.core[q], crank_q = sm.cpu_rank[q], grank_q = sm.gpu_rank[q];
#pragma unroll
      for (int s = 0; s < S; ++s)
        if (valid[s] && core_q == core[s] && crank_q < me.cpu_rank[s] && grank_q > gpu_rank[s]) broken = 1;
    }
    if (group_or<LPT>(broken, gmask)) {
#pragma unroll
      for (int s = 0; s < S; ++s)
        if (valid[s]) p.out_wcrt[a + lane + LPT * s] = GCAPS_WCRT_INVALID;
      if (lane == 0) p.out_sched[t] = GCAPS_SCHED_INVALID;
      return;
    }
    for (int i = 0; i < n; ++i) {
      const int rank_i = sm.gpu_rank[i];
      bool above[S];
#pragma unroll
      for (int s = 0; s < S; ++s) above[s] = gpu_rank[s] < rank_i;
      const i64 r = bound_at<LPT, S>(me, sm, i, above, fits32, busy, literal, lane, gmask);
      if (lane == 0) {
        p.out_wcrt[a + i] = r;
        if (g.gpu_prio_out) g.gpu_prio_out[a + i] = g.gpu_prio_in[a + i];
      }
      if (r < 0) sched = GCAPS_SCHED_NO;
    }
  } else {
    sched = search_levels<LPT, S>(g, a, n, me, core, valid, sm, fits32, busy, literal, lane, gmask);
  }
  if (lane == 0) p.out_sched[t] = (uint8_t)sched;
  __syncwarp(gmask);
}

// The search in integers for the kernel that holds search_narrow too: from global memory (a taskset that
// stage_fast declines), and from what stage_fast has left (one with a period of kNarrowLimit or more).
template <int LPT, int S>
__device__ __noinline__ void search_exact(const GpParams &g, i64 t, GpSmem<LPT * S> &sm, int lane, unsigned int gmask) {
  analyse_gpu_priority<LPT, S, true>(g, t, sm, lane, gmask);
}
template <int LPT, int S>
__device__ __noinline__ void search_wide(const GpParams &g, i64 t, i64 a, const TaskValues<S> &o, u32 *buf, int lane,
                                         unsigned int gmask) {
  const KParams &p = g.k;
  const bool busy = (p.policy & GCAPS_RTA_BUSY) != 0, literal = (p.policy & GCAPS_RTA_LITERAL) != 0;
  const Rows<LPT, S, false> rows{buf};
  GpSmem<LPT * S> &sm = *reinterpret_cast<GpSmem<LPT * S> *>(buf);
  u64 T[S], D[S], A[S], Ge[S], Star[S];
  int eta[S], core[S];
  bool valid[S];
  GpLane<S> me;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    valid[s] = lane + LPT * s < o.n;
    T[s] = 2, D[s] = 1, A[s] = 0, Ge[s] = 0, Star[s] = 0, eta[s] = 0, core[s] = -1, me.cpu_rank[s] = 0;
    if (valid[s]) {
      const uint4 row = rows.a(o.rank[s]);
      T[s] = o.T[s], D[s] = row.x, A[s] = o.A[s], Ge[s] = o.Ge[s], eta[s] = (int)o.eta[s], core[s] = (int)row.y;
      Star[s] = 2 * (u64)p.ovh * (u64)o.eta[s], me.cpu_rank[s] = o.rank[s];
    }
  }
  __syncwarp(gmask);  // (the rows are read: their place holds `sm` from here on)
#pragma unroll
  for (int s = 0; s < S; ++s)
    if (valid[s]) sm.core[lane + LPT * s] = core[s];
  lane_values<LPT, S>((u64)p.ovh, busy, true, T, D, A, Ge, Star, eta, core, valid, me, sm, lane);
  __syncwarp(gmask);
  const int sched = search_levels<LPT, S>(g, a, o.n, me, core, valid, sm, true, busy, literal, lane, gmask);
  if (lane == 0) p.out_sched[t] = (uint8_t)sched;
  __syncwarp(gmask);
}

// The search of Sec. 5.3 in single precision.  Called by the whole warp; its groups step from bound to
// bound side by side and sweep until the last of them has settled.  Returns, per group, whether its
// taskset is done (outputs written).
//
// Bound by instruction issue (4,204 warp instructions per 80-task taskset of `large`, 61 % of the issue
// slots; about 15 bounds and 43 sweeps each).  100,000 of them 1.19 -> 0.72 ms: what went are per-lane
// loops over global memory for the sums, a quadratic loop for every core's lowest task, 64-bit state
// and the integer form of the terms (7,230 instructions).
//
// DIRECT (a block of its own per taskset): prefetches, and searches a taskset with a longer period in
// integers; otherwise such a taskset is declined before its segments are read.
template <int LPT, int S, bool BUSY, bool DIRECT = false>
__device__ __forceinline__ bool search_narrow(const GpParams &g, bool live, i64 t, i64 a, int n, u32 *buf, int lane,
                                              unsigned int gmask) {
  const KParams &p = g.k;
  const bool literal = (p.policy & GCAPS_RTA_LITERAL) != 0;
  const u32 eps = (u32)p.ovh;
  const Rows<LPT, S, false> rows{buf};
  TaskValues<S> o;
  if (!stage_fast<LPT, S, (S <= 3 ? S : 2), true, DIRECT, !DIRECT>(p, live, a, n, buf, rows, lane, gmask, false, eps, o)) return false;
  live = o.live;
  if constexpr (DIRECT) {
    if (__any_sync(kFull, live && o.n_narrow != o.n)) {
      const TaskValues<S> there = o;  // (in memory for the call; `o` itself stays in registers)
      if (live) search_wide<LPT, S>(g, t, a, there, buf, lane, gmask);
      return live;
    }
  }
  n = o.n;
  // what this lane's tasks contribute as interferers; inv = 0 where there is no task
  float inv[S], Kc[S], Kg[S], Wc[S], We[S], Wes[S];
  u32 core[S], found[S];  // found: level << 23 | bound, 0 without a level
  PairConsts pc;
  pc.ovh = eps, pc.slot_cost = 0;
  u32 unplaced = 0;  // bit s: the task of slot s has no level yet
#pragma unroll
  for (int s = 0; s < S; ++s) {
    inv[s] = Kc[s] = Kg[s] = Wc[s] = We[s] = Wes[s] = 0.0f, core[s] = 0xffffffffu, found[s] = 0;
    if (lane + LPT * s < n) {
      uint4 row = rows.a(o.rank[s]);
      const float T = (float)o.T[s], D = (float)row.x, A = (float)o.A[s], Ge = (float)o.Ge[s];
      const bool gpu = o.eta[s] > 0;
      u32 star, base;
      own_cost<true>(pc, o.A[s], o.Ge[s], o.eta[s], 0, 0, star, base);
      // Sec. 6.4: J^c_h = D_h - (C_h + G^m_h), J^g_h = D_h - G^e_h (a task whose own execution exceeds
      // its deadline has no such slack: 0); a CPU-only tau_h has no J^c (Lemma 15), and none matters
      // in busy-waiting mode.  As J + T - 1/2 - 2^23, like in the recurrence.
      const float k = (T - 0.5f) - kTwo23, St = (float)star;
      inv[s] = __frcp_rn(T), core[s] = row.y;
      Kc[s] = (!BUSY && gpu) ? k + fmaxf(D - A, 0.0f) : k;
      Kg[s] = k + fmaxf(D - Ge, 0.0f);
      We[s] = Ge, Wes[s] = gpu ? Ge + St : 0.0f;
      Wc[s] = BUSY ? A : A + St;  // Lemma 12: C_h + G^m_h; Lemma 15: C_h + G^{m*}_h (star = 0 without segments)
      unplaced |= 1u << s;
      row.x += kOne23;
      row.z = kOne23 + (base < 0x7fffffu ? base : 0x7fffffu);
      row.w = (u32)(lane + LPT * s) | (gpu ? 0x10000u : 0u);
      rows.a(o.rank[s]) = row;
    }
  }
  __syncwarp();
  auto group_max = [&](int v) -> int {
    if constexpr (LPT == 32) {
      return __reduce_max_sync(kFull, v);
    } else {
#pragma unroll
      for (int d = 1; d < LPT; d <<= 1) {
        const int y = __shfl_xor_sync(kFull, v, d);
        v = y > v ? y : v;
      }
      return v;
    }
  };
  // cand: bit r set = the task of CPU rank r has no level yet and no task of lower CPU priority on its
  // core is without one, i.e. it may take the next level (the same-core rule of Sec. 5.3).  To start
  // with, the lowest task of every core.
  constexpr int kWords = LPT * S > 32 ? LPT * S / 32 : 1;
  u32 cand[kWords];
#pragma unroll
  for (int k = 0; k < kWords; ++k) cand[k] = 0;
  auto flip = [&](int r) {
#pragma unroll
    for (int k = 0; k < kWords; ++k)
      if (r >= 0 && (r >> 5) == k) cand[k] ^= 1u << (r & 31);
  };
  {
    u32 rest = unplaced;
#pragma unroll 1
    for (;;) {
      int low = -1;
#pragma unroll
      for (int s = 0; s < S; ++s)
        if ((rest >> s & 1u) && o.rank[s] > low) low = o.rank[s];
      low = group_max(low);
      if (LPT == 32 ? low < 0 : !__any_sync(kFull, low >= 0)) break;
      flip(low);
      const u32 its_core = rows.a(low < 0 ? 0 : low).y;
#pragma unroll
      for (int s = 0; s < S; ++s)
        if (core[s] == its_core) rest &= ~(1u << s);
      if (low < 0) rest = 0;
    }
  }
  bool active = live && n > 0;
  int sched = GCAPS_SCHED_YES, level = 1, want = n;
#pragma unroll 1
  for (;;) {
    // ---- the next candidate, from the lowest CPU priority upwards ---------------------------------
    int next = -1;
#pragma unroll
    for (int k = 0; k < kWords; ++k) {
      const int below = want - 32 * k;  // ranks 32 k .. 32 k + 31 that count: those below `want`
      const u32 m = below >= 32 ? cand[k] : (below <= 0 ? 0u : cand[k] & ((1u << below) - 1u));
      if (m) next = 32 * k + 31 - __clz((int)m);
    }
    want = next;
    if (active && want < 0) sched = GCAPS_SCHED_NO, active = false;
    if (LPT == 32 ? !active : !__any_sync(kFull, active)) break;
    const uint4 row = rows.a(want < 0 ? 0 : want);
    const u32 core_i = row.y;
    const float Db = __uint_as_float(row.x), base_b = __uint_as_float(row.z);
    const int c = (int)(row.w & 0xffffu);
    const bool gi = (row.w & 0x10000u) != 0;
    // ---- the (J, W) pairs; W = 0 where a pair does not apply ----------------------------------------
    f32x2 I2[S], J2[S], W2[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const bool hpp = core[s] == core_i && o.rank[s] < want;
      const bool hpg = (unplaced >> s & 1u) && !hpp && lane + LPT * s != c;  // hp(tau_i) of Sec. 6.4 minus hpp
      float w1 = 0.0f, w2 = 0.0f;
      if (BUSY) {
        if (hpp) w1 = Wc[s] + ((gi || !literal) ? Wes[s] : 0.0f);  // Lemmas 12, 10
        if (hpg) w2 = Wes[s];                                      // Lemmas 10, 11
      } else {
        if (hpp) w1 = Wc[s];                                       // Lemma 15
        if (gi) w2 = hpp ? We[s] : (hpg ? Wes[s] : 0.0f);          // Lemma 13: same core, other cores
      }
      I2[s] = pack2(inv[s], inv[s]), J2[s] = pack2(Kc[s], Kg[s]), W2[s] = pack2(w1, w2);
    }
    const f32x2 two23 = pack2(kTwo23, kTwo23), minus23 = pack2(-kTwo23, -kTwo23);
    const u32 base_bits = __float_as_uint(base_b) - 32u * kOne23;
    const f32x2 acc0 = LPT == 32 ? pack2(kTwo23, 0.0f) : pack2(0.0f, 0.0f);
    auto total = [&](f32x2 acc) -> float {  // base + the group's sum, as 2^23 + value
      float f = sum2(acc);
      if constexpr (LPT == 32) {
        f = fminf(f, kTwo23 + 4194304.0f);
        return __uint_as_float(__reduce_add_sync(kFull, __float_as_uint(f)) + base_bits);
      } else {
#pragma unroll
        for (int d = 1; d < LPT; d <<= 1) f += __shfl_xor_sync(kFull, f, d);
        return base_b + f;
      }
    };
    f32x2 acc = acc0;
#pragma unroll
    for (int s = 0; s < S; ++s) acc = add2(acc, W2[s]);
    const float all_once = total(acc);  // (a first iterate as in recurrence_narrow)
    float R = (Db - base_b < (float)GCAPS_RTA_ITER_CAP && base_b > kTwo23) ? all_once : base_b;
    bool go = active && !(R > Db);
    int left = (int)GCAPS_RTA_ITER_CAP;
#pragma unroll 1
    while ((LPT == 32 ? go : __any_sync(kFull, go)) && left > 0) {
      left -= 1;
      const f32x2 RR = pack2(R, R);
      acc = acc0;
#pragma unroll
      for (int s = 0; s < S; ++s) {
        const f32x2 q = fma2_down(add2(RR, J2[s]), I2[s], two23);
        acc = fma2(add2(q, minus23), W2[s], acc);
      }
      const float to = total(acc);
      const bool moved = go && to != R;
      R = moved ? to : R;
      go = moved && !(R > Db);
    }
    // ---- a bound within the deadline takes the level -------------------------------------------------
    const bool placed = active && !go && !(R > Db);
    if (LPT == 32 ? placed : __any_sync(kFull, placed)) {
      int up = -1;  // the task of the core that becomes a candidate now
#pragma unroll
      for (int s = 0; s < S; ++s) {
        if (placed && lane + LPT * s == c) {
          unplaced &= ~(1u << s);
          found[s] = ((u32)level << 23) | (__float_as_uint(R) - kOne23);
        }
        if ((unplaced >> s & 1u) && core[s] == core_i && o.rank[s] < want && o.rank[s] > up) up = o.rank[s];
      }
      up = group_max(up);
      if (placed) {
        flip(want);
        flip(up);
        level += 1, want = n;
        if (level > n) active = false;
      }
    }
  }
  // ---- results ------------------------------------------------------------------------------------------
#pragma unroll
  for (int s = 0; s < S; ++s) {
    if (lane + LPT * s < n) {
      const u32 lv = found[s] >> 23;
      p.out_wcrt[a + lane + LPT * s] = lv > 0 ? (i64)(found[s] & 0x7fffffu) : (i64)GCAPS_WCRT_MISS;
      g.gpu_prio_out[a + lane + LPT * s] = (i64)lv;
    }
  }
  if (live && lane == 0) p.out_sched[t] = (uint8_t)sched;
  __syncwarp();
  return live;
}

// The tasksets of one size bin, pulled in chunks from the bin's counter by the warps of the launch; the
// next chunk is looked up while the current one is worked on.  `warp_buf` is this warp's own shared
// memory (the same stride for every bin a kernel covers: the warps of a block may be working on
// different bins at the same time).
template <int LPT, int S, bool BUSY>
__device__ __forceinline__ void run_gp_bin(const GpParams &g, int bin, u32 *warp_buf, Ahead *ahead) {
  constexpr int G = 32 / LPT, MAXN = LPT * S;  // tasksets per warp
  typedef FastLayout<LPT, S> Lay;
  const KParams &p = g.k;
  const int lane32 = threadIdx.x & 31, group = lane32 / LPT, lane = lane32 % LPT;
  const unsigned int gmask = LPT == 32 ? kFull : (((1u << LPT) - 1u) << (group * LPT));
  u32 *const buf = warp_buf + group * Lay::kWords;
  const unsigned int start = p.hdr->bin_start[bin], count = p.hdr->bin_count[bin];
  if (count == 0) return;
  const bool fast_call = p.ovh < (1 << 20);
  unsigned int marked = 0;  // tasksets of this lane's group left to gpu_priority_rest_kernel
  const unsigned int n_groups = gridDim.x * (kBlockThreads / 32) * G;
  const int chunk = G * (count >= 32 * n_groups ? (G == 1 ? 8 : kMaxAhead / G) : (count >= 8 * n_groups ? 2 : 1));
  auto look_up = [&](unsigned int first, Ahead *slot) {
    if (lane32 < chunk)
      slot[lane32] = look_up_taskset<MAXN, Lay::CAP>(p, (first < count && first + lane32 < count) ? p.perm[start + first + lane32] : kNoTaskset);
    __syncwarp();
  };
  auto pull = [&]() {
    unsigned int first = 0;
    if (lane32 == 0) first = atomicAdd(&p.hdr->next[bin], (unsigned int)chunk);
    return __shfl_sync(kFull, first, 0);
  };
  unsigned int first = pull();
  int which = 0;
  look_up(first, ahead);
  while (first < count) {
    const unsigned int nfirst = pull();
    look_up(nfirst, ahead + (which ^ 1) * kMaxAhead);
    const Ahead *cur = ahead + which * kMaxAhead;
    const int in_chunk = count - first < (unsigned int)chunk ? (int)(count - first) : chunk;
#pragma unroll 1
    for (int c = 0; c < in_chunk; c += G) {
      const bool have = c + group < in_chunk;
      const Ahead me = cur[have ? c + group : 0];
      const bool fast = have && fast_call && (me.packed >> 31) != 0;
      bool done = false;
      if (fast_call) {
        if (fast) prefetch_segments<LPT>(p, me, lane);
        done = search_narrow<LPT, S, BUSY>(g, fast, (i64)me.t, me.a, (int)(me.packed & 0x1ffu), buf, lane, gmask);
      }
      __syncwarp();
      if (have && !done && lane == 0) p.perm[start + first + c + group] |= kDeferred, marked += 1;
      __syncwarp();
    }
    first = nfirst;
    which ^= 1;
  }
  if (marked > 0) atomicAdd(&p.hdr->deferred[bin], marked);
}

// What run_gp_bin has marked in a bin: tasksets with a period of kNarrowLimit or more, values beyond the 32-bit
// path, malformed ones.  Where most of the bin is marked its entries are pulled from a counter, as many as
// the warp has groups; where few are, every warp looks through its share, 32 entries at a time.
template <int LPT, int S>
__device__ __forceinline__ void run_rest_bin(const GpParams &g, int bin, unsigned char *warp_smem) {
  constexpr unsigned int G = 32 / LPT;
  typedef GpSmem<LPT * S> Sm;
  const KParams &p = g.k;
  const unsigned int lane32 = threadIdx.x & 31, group = lane32 / LPT;
  const int lane = (int)(lane32 % LPT);
  const unsigned int gmask = LPT == 32 ? kFull : (((1u << LPT) - 1u) << (group * LPT));
  const unsigned int start = p.hdr->bin_start[bin], count = p.hdr->bin_count[bin];
  const unsigned int marked = count > 0 ? __ldcg(&p.hdr->deferred[bin]) : 0;
  if (marked == 0) return;
  const bool dense = marked >= count / 4;
  const unsigned int n_warps = gridDim.x * (kBlockThreads / 32), step = dense ? G : 32;
  unsigned int window = (blockIdx.x * (kBlockThreads / 32) + (threadIdx.x >> 5)) * 32;  // (!dense)
  for (;;) {
    unsigned int first = window;
    if (dense) {
      if (lane32 == 0) first = atomicAdd(&p.hdr->next2[bin], step);
      first = __shfl_sync(kFull, first, 0);
    }
    window += n_warps * 32;
    if (first >= count) break;
    u32 t = 0;
    if (lane32 < step && first + lane32 < count) t = __ldcg(&p.perm[start + first + lane32]);
    unsigned int found = __ballot_sync(kFull, (t & kDeferred) != 0);
    while (found) {  // the next G of them, one per group
      unsigned int rest = found;
      for (unsigned int k = 0; k < group; ++k) rest &= rest - 1;
      const bool have = rest != 0;
      const u32 mine = __shfl_sync(kFull, t, have ? __ffs((int)rest) - 1 : 0) & ~kDeferred;
      if (have) analyse_gpu_priority<LPT, S, true>(g, (i64)mine, reinterpret_cast<Sm *>(warp_smem)[group], lane, gmask);
      __syncwarp();
      for (unsigned int k = 0; k < G; ++k) found &= found - 1;
    }
  }
}

// the four bins of up to 32 tasks: (lanes per taskset, tasks per lane) as in the default analysis
template <bool BUSY>
__global__ void __launch_bounds__(kBlockThreads, 5) gpu_priority_small_kernel(GpParams g) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  let_dependents_start();  // the kernel of the next size bin shares no data with this one
  u32 *mine = reinterpret_cast<u32 *>(smem_raw) + (threadIdx.x >> 5) * kSmallWarpWords;
  Ahead *ahead = reinterpret_cast<Ahead *>(mine + kSmallWarpWords - kAheadWords);
  run_gp_bin<16, 2, BUSY>(g, 3, mine, ahead);
  run_gp_bin<8, 3, BUSY>(g, 2, mine, ahead);
  run_gp_bin<8, 2, BUSY>(g, 1, mine, ahead);
  run_gp_bin<8, 1, BUSY>(g, 0, mine, ahead);
  wait_for_previous_grid();
}

// one bin of larger tasksets, a warp per taskset
__host__ __device__ constexpr int gp_min_blocks(int slots) { return slots <= 3 ? 5 : slots == 4 ? 4 : 2; }
template <int S, bool BUSY>
__global__ void __launch_bounds__(kBlockThreads, gp_min_blocks(S)) gpu_priority_big_kernel(GpParams g, int bin) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  let_dependents_start();
  constexpr int kWarpWords = bin_warp_words<32, S>() + kAheadWords;
  u32 *mine = reinterpret_cast<u32 *>(smem_raw) + (threadIdx.x >> 5) * kWarpWords;
  run_gp_bin<32, S, BUSY>(g, bin, mine, reinterpret_cast<Ahead *>(mine + kWarpWords - kAheadWords));
  wait_for_previous_grid();
}

// A batch of at most kDirectSweepMost tasksets in one launch: a block of one warp per taskset, no plan
// (1,000 tasksets of 8 / 20 / 80 tasks: 25 / 26 / 45 us, with plan and binned kernels 39 / 59 / 66 us; 4,096
// of them: 36 / 60 / 87 against 40 / 65 / 88 us, and 313 against 250 us where all 80 tasks find a level).
template <int S, bool BUSY>
__device__ __forceinline__ void search_direct(const GpParams &g, bool fast, i64 t, i64 a, int n, u32 *buf, int lane) {
  const bool done = fast && search_narrow<32, S, BUSY, true>(g, true, t, a, n, buf, lane, kFull);
  __syncwarp();
  if (!done) search_exact<32, S>(g, t, *reinterpret_cast<GpSmem<32 * S> *>(buf), lane, kFull);
}
template <bool BUSY>
__global__ void __launch_bounds__(32) gpu_priority_direct_kernel(GpParams g) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  u32 *const buf = reinterpret_cast<u32 *>(smem_raw);
  const KParams &p = g.k;
  const int lane = threadIdx.x;
  const i64 t = blockIdx.x;
  const i64 a = p.task_off[t], b = p.task_off[t + 1];
  // (a broken range goes to the exact search of the smallest size, which finds it INVALID)
  const bool in_range = a >= 0 && b > a && b <= p.n_tasks && b - a <= GCAPS_RTA_MAX_TASKS;
  const bool fast = in_range && p.ovh < (1 << 20);
  const int n = in_range ? (int)(b - a) : 0;
  if (n <= 32) search_direct<1, BUSY>(g, fast, t, a, n, buf, lane);
  else if (n <= 64) search_direct<2, BUSY>(g, fast, t, a, n, buf, lane);
  else if (n <= 96) search_direct<3, BUSY>(g, fast, t, a, n, buf, lane);
  else if (n <= 128) search_direct<4, BUSY>(g, fast, t, a, n, buf, lane);
  else if (n <= 192) search_direct<6, BUSY>(g, fast, t, a, n, buf, lane);
  else search_direct<8, BUSY>(g, fast, t, a, n, buf, lane);
}

// Given GPU priorities: every task is bounded once, in integers.
template <int LPT, int S>
__device__ __forceinline__ void run_given_bin(const GpParams &g, int bin, unsigned char *warp_smem) {
  constexpr int G = 32 / LPT;  // tasksets per warp
  typedef GpSmem<LPT * S> Sm;
  const KParams &p = g.k;
  const int lane32 = threadIdx.x & 31, group = lane32 / LPT, lane = lane32 % LPT;
  const unsigned int gmask = LPT == 32 ? kFull : (((1u << LPT) - 1u) << (group * LPT));
  const unsigned int start = p.hdr->bin_start[bin], count = p.hdr->bin_count[bin];
  for (;;) {
    unsigned int first = 0;
    if (lane32 == 0) first = atomicAdd(&p.hdr->next[bin], (unsigned int)G);
    first = __shfl_sync(kFull, first, 0);
    if (first >= count) break;
    if (first + group < count)
      analyse_gpu_priority<LPT, S, false>(g, (i64)p.perm[start + first + group], reinterpret_cast<Sm *>(warp_smem)[group],
                                          lane, gmask);
    __syncwarp();
  }
}
template <int LPT, int S>
__host__ __device__ constexpr int given_warp_bytes() {
  return (32 / LPT) * (int)sizeof(GpSmem<LPT * S>);
}
constexpr int kGivenSmallWarpBytes = cmax(cmax(given_warp_bytes<16, 2>(), given_warp_bytes<8, 3>()),
                                          cmax(given_warp_bytes<8, 2>(), given_warp_bytes<8, 1>()));
static_assert(kGivenSmallWarpBytes % 16 == 0, "every warp's area starts 16-byte aligned");
__global__ void __launch_bounds__(kBlockThreads) gpu_priority_given_small_kernel(GpParams g) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  let_dependents_start();
  unsigned char *mine = smem_raw + (threadIdx.x >> 5) * kGivenSmallWarpBytes;
  run_given_bin<16, 2>(g, 3, mine);
  run_given_bin<8, 3>(g, 2, mine);
  run_given_bin<8, 2>(g, 1, mine);
  run_given_bin<8, 1>(g, 0, mine);
  wait_for_previous_grid();
}
template <int S>
__global__ void __launch_bounds__(kBlockThreads, S <= 4 ? 5 : 2) gpu_priority_given_big_kernel(GpParams g, int bin) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  let_dependents_start();
  run_given_bin<32, S>(g, bin, smem_raw + (threadIdx.x >> 5) * given_warp_bytes<32, S>());
  wait_for_previous_grid();
}
// ... of a batch of at most kDirectGivenMost tasksets, a block of one warp per taskset, without a plan: 1,000
// tasksets of 8 / 20 / 80 / 128 tasks 24 / 27 / 113 / 196 us, with plan and binned kernels 40 / 63 / 155 / 280
// us; 4,096 of them 36 / 72 / 359 / 615 against 53 / 86 / 274 / 508 us.
__global__ void __launch_bounds__(32) gpu_priority_given_direct_kernel(GpParams g) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const KParams &p = g.k;
  const int lane = threadIdx.x;
  const i64 t = blockIdx.x, n = p.task_off[t + 1] - p.task_off[t];
  // (a broken range is found INVALID whatever its size)
  if (n <= 32) analyse_gpu_priority<32, 1, false>(g, t, *reinterpret_cast<GpSmem<32> *>(smem_raw), lane, kFull);
  else if (n <= 64) analyse_gpu_priority<32, 2, false>(g, t, *reinterpret_cast<GpSmem<64> *>(smem_raw), lane, kFull);
  else if (n <= 96) analyse_gpu_priority<32, 3, false>(g, t, *reinterpret_cast<GpSmem<96> *>(smem_raw), lane, kFull);
  else if (n <= 128) analyse_gpu_priority<32, 4, false>(g, t, *reinterpret_cast<GpSmem<128> *>(smem_raw), lane, kFull);
  else if (n <= 192) analyse_gpu_priority<32, 6, false>(g, t, *reinterpret_cast<GpSmem<192> *>(smem_raw), lane, kFull);
  else analyse_gpu_priority<32, 8, false>(g, t, *reinterpret_cast<GpSmem<256> *>(smem_raw), lane, kFull);
}

// What the search's kernels have left over, largest tasksets first (100,000 tasksets of 20 tasks with periods
// to 60 s: 572 us; out of line in those kernels 762, without the look at them first 520).
constexpr int kRestWarpBytes = cmax(given_warp_bytes<32, 8>(), kGivenSmallWarpBytes);
static_assert(kRestWarpBytes % 16 == 0, "every warp's area starts 16-byte aligned");
__global__ void __launch_bounds__(kBlockThreads, 4) gpu_priority_rest_kernel(GpParams g) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  wait_for_previous_grid();  // the marks in the permutation are complete from here on
  unsigned char *mine = smem_raw + (threadIdx.x >> 5) * kRestWarpBytes;
  run_rest_bin<32, 8>(g, 8, mine);
  run_rest_bin<32, 6>(g, 7, mine);
  run_rest_bin<32, 4>(g, 6, mine);
  run_rest_bin<32, 3>(g, 5, mine);
  run_rest_bin<32, 2>(g, 4, mine);
  run_rest_bin<16, 2>(g, 3, mine);
  run_rest_bin<8, 3>(g, 2, mine);
  run_rest_bin<8, 2>(g, 1, mine);
  run_rest_bin<8, 1>(g, 0, mine);
}

template <int S, bool BUSY>
cudaError_t launch_big(const GpParams &g, int bin, int sm_count, cudaStream_t st) {
  constexpr int kWarps = kBlockThreads / 32;
  static int blocks_per_sm[64] = {0};
  return launch_persistent_ex(true, gpu_priority_big_kernel<S, BUSY>, blocks_per_sm,
                              sizeof(u32) * (bin_warp_words<32, S>() + kAheadWords) * kWarps,
                              (g.k.n_tasksets + kWarps - 1) / kWarps, sm_count, st, g, bin);
}

template <bool BUSY>
cudaError_t launch_gp_bins(const GpParams &g, int sm_count, cudaStream_t st) {
  constexpr int kWarps = kBlockThreads / 32;
  static int blocks_per_sm[64] = {0};
  cudaError_t e = launch_persistent(gpu_priority_small_kernel<BUSY>, blocks_per_sm, sizeof(u32) * kSmallWarpWords * kWarps,
                                    (g.k.n_tasksets + kWarps - 1) / kWarps, sm_count, st, g);
  if (e == cudaSuccess) e = launch_big<2, BUSY>(g, 4, sm_count, st);
  if (e == cudaSuccess) e = launch_big<3, BUSY>(g, 5, sm_count, st);
  if (e == cudaSuccess) e = launch_big<4, BUSY>(g, 6, sm_count, st);
  if (e == cudaSuccess) e = launch_big<6, BUSY>(g, 7, sm_count, st);
  if (e == cudaSuccess) e = launch_big<8, BUSY>(g, 8, sm_count, st);
  static int rest_blocks_per_sm[64] = {0};
  if (e == cudaSuccess)
    e = launch_persistent_ex(true, gpu_priority_rest_kernel, rest_blocks_per_sm, (size_t)kRestWarpBytes * kWarps,
                             (g.k.n_tasksets + kWarps - 1) / kWarps, sm_count, st, g);
  return e;
}

template <int S>
cudaError_t launch_given_big(const GpParams &g, int bin, int sm_count, cudaStream_t st) {
  constexpr int kWarps = kBlockThreads / 32;
  static int blocks_per_sm[64] = {0};
  return launch_persistent_ex(true, gpu_priority_given_big_kernel<S>, blocks_per_sm, (size_t)given_warp_bytes<32, S>() * kWarps,
                              (g.k.n_tasksets + kWarps - 1) / kWarps, sm_count, st, g, bin);
}

cudaError_t launch_given_bins(const GpParams &g, int sm_count, cudaStream_t st) {
  constexpr int kWarps = kBlockThreads / 32;
  static int blocks_per_sm[64] = {0};
  cudaError_t e = launch_persistent(gpu_priority_given_small_kernel, blocks_per_sm, (size_t)kGivenSmallWarpBytes * kWarps,
                                    (g.k.n_tasksets + kWarps - 1) / kWarps, sm_count, st, g);
  if (e == cudaSuccess) e = launch_given_big<2>(g, 4, sm_count, st);
  if (e == cudaSuccess) e = launch_given_big<3>(g, 5, sm_count, st);
  if (e == cudaSuccess) e = launch_given_big<4>(g, 6, sm_count, st);
  if (e == cudaSuccess) e = launch_given_big<6>(g, 7, sm_count, st);
  if (e == cudaSuccess) e = launch_given_big<8>(g, 8, sm_count, st);
  return e;
}

}  // namespace

extern "C" int gcaps_rta_gpu_priority_batch(const gcaps_tasksets_t *ts, int64_t n_tasksets, int flags,
                                            int64_t runlist_update_us, const int64_t *gpu_priority,
                                            int64_t *out_gpu_priority, int64_t *out_wcrt,
                                            uint8_t *out_sched, void *workspace,
                                            size_t workspace_bytes, void *stream) {
  if (flags & ~(GCAPS_RTA_BUSY | GCAPS_RTA_LITERAL | GCAPS_RTA_ASSIGN)) return GCAPS_ERR_INVALID_ARG;
  const int policy = GCAPS_POLICY_GCAPS | (flags & (GCAPS_RTA_BUSY | GCAPS_RTA_LITERAL));
  int rc = check_args(ts, n_tasksets, policy, 1, runlist_update_us);
  if (rc != GCAPS_OK) return rc;
  const bool assign = (flags & GCAPS_RTA_ASSIGN) != 0;
  if (n_tasksets == 0) return GCAPS_OK;
  if (!out_sched || (ts->n_tasks > 0 && (!out_wcrt || (assign ? !out_gpu_priority : !gpu_priority))))
    return GCAPS_ERR_INVALID_ARG;
  DeviceInfo di;
  rc = device_info(&di);
  if (rc != GCAPS_OK) return rc;
  GpParams g;
  fill_params(&g.k, ts, n_tasksets, policy, 1, runlist_update_us, out_wcrt, out_sched);
  g.gpu_prio_in = (const i64 *)gpu_priority;
  g.gpu_prio_out = (i64 *)out_gpu_priority;
  cudaStream_t st = (cudaStream_t)stream;
  const bool direct = n_tasksets <= (assign ? kDirectSweepMost : kDirectGivenMost), busy = (flags & GCAPS_RTA_BUSY) != 0;
  rc = direct ? place_plan(g.k, workspace, workspace_bytes) : enqueue_plan(g.k, workspace, workspace_bytes, st);
  if (rc != GCAPS_OK) return rc;
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess && direct) {
    constexpr int smem = (int)sizeof(u32) * bin_warp_words<32, 8>();
    static_assert(sizeof(GpSmem<256>) <= (size_t)smem && smem <= 48 * 1024, "no attribute to set");
    if (!assign) gpu_priority_given_direct_kernel<<<(unsigned int)n_tasksets, 32, sizeof(GpSmem<256>), st>>>(g);
    else if (busy) gpu_priority_direct_kernel<true><<<(unsigned int)n_tasksets, 32, smem, st>>>(g);
    else gpu_priority_direct_kernel<false><<<(unsigned int)n_tasksets, 32, smem, st>>>(g);
    e = cudaGetLastError();
  } else if (e == cudaSuccess && !assign) {
    e = launch_given_bins(g, di.sm_count, st);
  } else if (e == cudaSuccess) {
    e = busy ? launch_gp_bins<true>(g, di.sm_count, st) : launch_gp_bins<false>(g, di.sm_count, st);
  }
  if (e != cudaSuccess) {
    g_last_cuda_error = (int)e;
    return GCAPS_ERR_CUDA;
  }
  return GCAPS_OK;
}
