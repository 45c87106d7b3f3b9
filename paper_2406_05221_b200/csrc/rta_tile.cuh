// rta_tile.cuh -- tasksets of up to 24 tasks, a tile of up to 32 of them per warp.  Internal.
//
//   stage   four tasksets at a time, eight lanes each: values are checked, the segments added up, and every
//           task's values go to the row of its position
//   order   lane = taskset from here on: positions by rank, positions by core
//   walk    every lane takes its own taskset through the recurrence, rank by rank, out of its column of
//           the tile, and writes its results.  Nothing is exchanged between lanes
//
// What bounds it.  With a group of lanes per taskset (run_bin) a 20-task taskset took 1,345 warp instructions: a
// sweep over its 10 interferers is one or two terms per lane and then a reduction, a vote and a branch, and setting
// a rank up is done by every group for itself.  A lane per taskset needs none of that: 669 instructions, though
// the lanes wait for the one with the most sweeps (123 in 20 ranks against 81 with four tasksets per warp, 53 for
// one alone).  What is left is latency: a tile of 20 ranks takes 24 KB, so an SM holds nine warps (eight on average).  Everything follows from
// that: interferers lie in registers, and a sweep is straight-line code for a bound on their number that the warp
// shares (2, 4 or 6 on the same core and twice as many in the list; with a branch per pair of entries the walk took
// 76,000 instead of 50,000 cycles per tile); a lane's stage has all loads of a task under way at once, out of L2.
// Two or four lanes per taskset, or copying the tasksets into shared memory first, were slower.  And as tiles take the
// batch in its order, there is no plan and there are no bins: five operations in the stream (the header is cleared; the tiles; the rest
// of a plan, for a batch that turns out to be none for tiles; two launches over what is left) instead of eleven.  100,000
// tasksets of 20 tasks at U/core 0.5 under GCAPS 226 -> 175 us (U/core 0.3 196 -> 146), under RR 133 -> 92; 1,000,000 of
// 8 tasks 634 -> 338 us; 200,000 of 24 tasks under RR 208 -> 157 us.
#ifndef GCAPS_RTA_TILE_CUH_
#define GCAPS_RTA_TILE_CUH_

#include <cuda_runtime.h>
#include <stdint.h>

#include "rta_device.cuh"
#include "tile_patience.h"

namespace {

constexpr int kTileThreads = 32;
constexpr int kTileMost = 24;      // tasks
constexpr int kTileSweeps = 4096;  // sweeps of a rank after which a taskset is left over
constexpr int kTileCores = 16;     // cores are 0 .. kTileCores-1
constexpr int kTileOnCore = 10;    // a walk is good for that many tasks of a core: it holds six of them in registers
constexpr int kTileGroup = 8;      // lanes per taskset in the stage

constexpr int kTileStride = 33;  // columns of a row: one more than tasksets, as the stage writes them with lanes at
                                 // different rows of one column
__host__ __device__ constexpr int tile_list_pairs(int rows) { return (rows + 3) / 4 * 2; }
// T, GPU segments and core of a task in one word
__device__ __forceinline__ u32 tile_word(u32 T, u32 gpu_segments, u32 core) { return T | gpu_segments << 22 | core << 28; }
__device__ __forceinline__ float tile_period(u32 word) { return (float)(word & 0x3fffffu); }
__device__ __forceinline__ u32 tile_segments(u32 word) { return (word >> 22) & 63u; }

// Shared memory of one warp's tile where every taskset is analysed once: rows by position, a column per taskset.  There is room for `rows`
// positions of 32 tasksets.
//   e4  before the task is bounded  T and more, D, A = C+G^m, G^e with the sign bit = uses the GPU
//       after                       1/T, J^c, W^c, J^g (GCAPS) or S (RR)
//   m   priority; after             S or W^g (GCAPS)
//   s   (RR) S
//   ord by rank: position
//   on_core  by core: positions (bits)
//   list (GCAPS)  the GPU-using tasks in rank order: 1/T, J^g, W^g, two entries side by side
template <int MODE>
struct TileRows {
  uint4 *e4;
  u32 *m, *s, *cores;
  f32x2 *g_inv, *g_j, *g_w;
  unsigned char *ord;
  int lane, list_pairs;

  static constexpr int kSets = 32;
  static __host__ __device__ constexpr int bytes(int rows) {
    return (rows * kTileStride * (MODE < 2 ? 20 : 24) + 15) / 16 * 16 + rows * 32 + kTileCores * 128 +
           (MODE < 2 ? tile_list_pairs(rows) * 32 * 24 : 0);
  }
  __device__ __forceinline__ TileRows(unsigned char *mem, int rows) {
    const int all = rows * kTileStride;
    lane = threadIdx.x & 31, list_pairs = tile_list_pairs(rows);
    e4 = reinterpret_cast<uint4 *>(mem);
    m = reinterpret_cast<u32 *>(mem + all * 16);
    s = MODE < 2 ? nullptr : reinterpret_cast<u32 *>(mem + all * 20);
    unsigned char *at = mem + (all * (MODE < 2 ? 20 : 24) + 15) / 16 * 16;
    cores = reinterpret_cast<u32 *>(at);
    ord = at + kTileCores * 128;
    const int plane = list_pairs * 32;
    g_inv = reinterpret_cast<f32x2 *>(ord + rows * 32);
    g_j = g_inv + plane, g_w = g_j + plane;
  }
  __device__ __forceinline__ void keep(const KParams &p, int i, int c, u32 T, u32 D, u32 core, u32 segments, u32, u32 A,
                                       u32 Ge, u32 slices, int priority) const {
    const int at = i * kTileStride + c;
    e4[at] = make_uint4(tile_word(T, segments, core), __float_as_uint((float)D), __float_as_uint((float)A),
                        __float_as_uint((float)Ge) | (segments > 0 ? 0x80000000u : 0u));
    m[at] = (u32)priority;
    if (MODE >= 2) {
      const u64 cost = (u64)p.L + (u64)p.ovh;
      const u64 S = slices == 0 ? 0 : (cost >= kFastClamp ? kFastClamp : cost * (u64)slices);
      s[at] = __float_as_uint((float)(u32)(S < kFastClamp ? S : kFastClamp));
    }
  }
  __device__ __forceinline__ i64 most_gsegs() const { return 64 * 32; }  // one more than a taskset may have
  __device__ __forceinline__ void keep_segment(int, u32, u32) const {}
  __device__ __forceinline__ int priority(int i) const { return (int)m[i * kTileStride + lane]; }
  __device__ __forceinline__ u32 word(int i) const { return e4[i * kTileStride + lane].x; }
  __device__ __forceinline__ uint4 own(int i) const { return e4[i * kTileStride + lane]; }
  __device__ __forceinline__ u32 &on_core(u32 core) const { return cores[core * 32 + lane]; }
  __device__ __forceinline__ unsigned char &order(int r) const { return ord[r * 32 + lane]; }
  __device__ __forceinline__ float slot_time(int i, const uint4 &, bool) const { return __uint_as_float(s[i * kTileStride + lane]); }
  // before the first rank
  __device__ __forceinline__ void clear() const {
    if (MODE < 2)
      for (int x = lane; x < list_pairs * 32; x += 32) g_inv[x] = g_j[x] = g_w[x] = pack2(0.0f, 0.0f);
  }
  // an entry of the same core: 1/T, J^c, W^c, J^g, and S or W^g
  template <class Mode>
  __device__ __forceinline__ void gcaps_core(Mode, int h, float, float &inv, float &jc, float &wc, float &jg, float &wg) const {
    const uint4 e = e4[h * kTileStride + lane];
    inv = __uint_as_float(e.x), jc = __uint_as_float(e.y), wc = __uint_as_float(e.z), jg = __uint_as_float(e.w);
    wg = __uint_as_float(m[h * kTileStride + lane]);
  }
  __device__ __forceinline__ void rr_core(int h, float &inv, float &j, float &A, float &S) const {
    const uint4 e = e4[h * kTileStride + lane];
    inv = __uint_as_float(e.x), j = __uint_as_float(e.y), A = __uint_as_float(e.z), S = __uint_as_float(e.w);
  }
  // entries 2q and 2q+1 of the list (behind its end: zeros)
  __device__ __forceinline__ void list(int q, int, float, f32x2 &I, f32x2 &J, f32x2 &W) const {
    const int x = (q < list_pairs ? q : 0) * 32 + lane;
    I = g_inv[x], J = g_j[x], W = g_w[x];
    if (q >= list_pairs) I = W = pack2(0.0f, 0.0f);
  }
  __device__ __forceinline__ void gcaps_publish(int i, float inv, float jc, float wc, float jg, float wg) const {
    const int at = i * kTileStride + lane;
    e4[at] = make_uint4(__float_as_uint(inv), __float_as_uint(jc), __float_as_uint(wc), __float_as_uint(jg));
    m[at] = __float_as_uint(wg);
  }
  __device__ __forceinline__ void rr_publish(int i, float inv, float j, float A, float S) const {
    e4[i * kTileStride + lane] = make_uint4(__float_as_uint(inv), __float_as_uint(j), __float_as_uint(A), __float_as_uint(S));
  }
  __device__ __forceinline__ void append(int k, int, float inv, float jg, float w) const {
    const int x = ((k >> 1) * 32 + lane) * 2 + (k & 1);
    reinterpret_cast<float *>(g_inv)[x] = inv, reinterpret_cast<float *>(g_j)[x] = jg, reinterpret_cast<float *>(g_w)[x] = w;
  }
};

// What lane c knows of the taskset of column c.
struct TileLane {
  i64 a, c, g;  // first task, first CPU segment, first GPU segment
  u32 t;        // taskset index
  int n;        // tasks; 0: no taskset, or one that the tile does not take
  int size;     // tasks all the same; 0: not 1 .. 256
  u32 nc, ng;   // segments
  bool declined;
};

// The tasks of columns c0 .. c0+3 go to their rows, U tasks per lane side by side.
// What is kept of a task: rows.keep(position, column, T, D, core, GPU segments, the first one, C+G^m, G^e, slices of Eq. 3, priority);
// SLICES: they are wanted.
template <int U, bool SLICES, class Rows>
__device__ __forceinline__ void tile_stage(const KParams &p, const Rows &rows, TileLane &me, int c0, int lane) {
  const int c = c0 + lane / kTileGroup, from = c & 31;
  const int n = __shfl_sync(kFull, me.n, from);
  const i64 a = __shfl_sync(kFull, me.a, from), cf = __shfl_sync(kFull, me.c, from), gf = __shfl_sync(kFull, me.g, from);
  const u32 nc = __shfl_sync(kFull, me.nc, from), ng = __shfl_sync(kFull, me.ng, from);
  auto slices_of = [&](u32 y) -> u32 {  // Eq. 3
    if (p.l_mode == 0) return __umulhi((y & (kFastLimit - 1)) + (u32)p.L - 1u, p.l_magic) >> p.l_shift;
    return p.l_mode == 1 ? y : (y > 0 ? 1u : 0u);
  };
  u32 bad = 0;
#pragma unroll 1
  for (int i0 = 0; __any_sync(kFull, i0 < n); i0 += U * kTileGroup) {
    u32 T[U], D[U], K[U], cn[U], gn[U], rc[U], rg[U], A[U], Ge[U], slices[U];
    int P[U];
    {
      i64 c64[U], c_end[U], g64[U], g_end[U], T64[U], D64[U], P64[U], K64[U];
      const i64 k = a + i0 + lane % kTileGroup;
      const i64 *const pT = p.period + k, *const pD = p.deadline + k, *const pP = p.priority + k, *const pK = p.core + k;
      const i64 *const pc = p.cseg_off + k, *const pg = p.gseg_off + k;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        c64[u] = c_end[u] = cf + p.cseg_base, g64[u] = g_end[u] = gf + p.gseg_base;
        T64[u] = 2, D64[u] = 1, P64[u] = K64[u] = 0;
        if (i0 + lane % kTileGroup + u * kTileGroup < n) {
          c64[u] = pc[u * kTileGroup], c_end[u] = pc[u * kTileGroup + 1], g64[u] = pg[u * kTileGroup], g_end[u] = pg[u * kTileGroup + 1];
          T64[u] = pT[u * kTileGroup], D64[u] = pD[u * kTileGroup], P64[u] = pP[u * kTileGroup], K64[u] = pK[u * kTileGroup];
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        // offsets relative to the taskset's first ones (its slices lie inside the arrays)
        const i64 r1 = c64[u] - p.cseg_base - cf, r2 = g64[u] - p.gseg_base - gf, d1 = c_end[u] - c64[u], d2 = g_end[u] - g64[u];
        u32 not_ok = (u32)((u64)r1 >> 32) | (u32)((u64)r2 >> 32) | (u32)((u64)d1 >> 32) | (u32)((u64)d2 >> 32);
        not_ok |= ((u32)d1 | (u32)d2) >> 6;
        rc[u] = (u32)r1, rg[u] = (u32)r2, cn[u] = (u32)d1, gn[u] = (u32)d2;
        not_ok |= rc[u] <= nc && cn[u] <= nc - rc[u] && rg[u] <= ng && gn[u] <= ng - rg[u] ? 0u : 1u;
        if (not_ok != 0) cn[u] = gn[u] = 0;
        T[u] = (u32)T64[u], D[u] = (u32)D64[u], K[u] = (u32)K64[u], P[u] = (int)P64[u];
        not_ok |= (u32)((u64)T64[u] >> 32) | (u32)((u64)D64[u] >> 32) | (u32)((u64)K64[u] >> 32);
        not_ok |= (u32)((u64)P64[u] >> 32) ^ (u32)(P[u] >> 31);
        not_ok |= K[u] / kTileCores;
        // 2 <= T < kNarrowLimit, 1 <= D <= T
        not_ok |= T[u] - 2u < kNarrowLimit - 2u && D[u] - 1u < T[u] ? 0u : 1u;
        bad |= not_ok;
      }
    }
    const i64 *const xc = p.cseg_wcet + cf, *const xm = p.gseg_misc + gf, *const xe = p.gseg_exec + gf;
    // four CPU and three GPU segments of every task side by side
    {
      i64 w[U][4], m[U][3], e[U][3];
#pragma unroll
      for (int u = 0; u < U; ++u) {
#pragma unroll
        for (u32 j = 0; j < 4; ++j) {
          w[u][j] = 0;
          if (j < cn[u]) w[u][j] = __ldg(xc + rc[u] + j);
        }
#pragma unroll
        for (u32 j = 0; j < 3; ++j) {
          m[u][j] = e[u][j] = 0;
          if (j < gn[u]) m[u][j] = __ldg(xm + rg[u] + j), e[u][j] = __ldg(xe + rg[u] + j);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const u64 all = ((u64)w[u][0] | (u64)w[u][1]) | ((u64)w[u][2] | (u64)w[u][3]) | ((u64)m[u][0] | (u64)m[u][1]) |
                        ((u64)m[u][2] | (u64)e[u][0]) | ((u64)e[u][1] | (u64)e[u][2]);
        bad |= (u32)(all >> 32) | ((u32)all >> 26);
        A[u] = ((u32)w[u][0] + (u32)w[u][1]) + ((u32)w[u][2] + (u32)w[u][3]) + ((u32)m[u][0] + (u32)m[u][1]) + (u32)m[u][2];
        Ge[u] = (u32)e[u][0] + (u32)e[u][1] + (u32)e[u][2];
        bad |= (A[u] | Ge[u]) >> 26;  // seven values below 2^26 do not wrap, nor does a sum below 2^26 with one or two more
#pragma unroll
        for (u32 j = 0; j < 3; ++j)
          if (j < gn[u]) rows.keep_segment(c, rg[u] + j, (u32)e[u][j]);
        slices[u] = SLICES ? slices_of((u32)e[u][0]) + slices_of((u32)e[u][1]) + slices_of((u32)e[u][2]) : 0u;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll 1
      for (u32 j = 4; j < cn[u]; ++j) {
        const u64 w = (u64)__ldg(xc + rc[u] + j);
        A[u] += (u32)w;
        bad |= (u32)(w >> 32) | (((u32)w | A[u]) >> 26);
      }
#pragma unroll 1
      for (u32 j = 3; j < gn[u]; ++j) {
        const u64 m = (u64)__ldg(xm + rg[u] + j), e = (u64)__ldg(xe + rg[u] + j);
        A[u] += (u32)m, Ge[u] += (u32)e;
        bad |= (u32)((m | e) >> 32) | (((u32)(m | e) | A[u] | Ge[u]) >> 26);
        rows.keep_segment(c, rg[u] + j, (u32)e);
        if (SLICES) slices[u] += slices_of((u32)e);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + lane % kTileGroup + u * kTileGroup;
      if (i < n) rows.keep(p, i, c, T[u], D[u], K[u], gn[u], rg[u], A[u], Ge[u], slices[u], P[u]);
    }
  }
  const u32 bad_bits = __ballot_sync(kFull, bad != 0);
  const u32 mine = (u32)(lane - c0);  // the lane of a column
  if (mine < 32 / kTileGroup && ((bad_bits >> (mine * kTileGroup)) & ((1u << kTileGroup) - 1u)) != 0) {
    if (me.n > 0) me.declined = true;
    me.n = 0;
  }
}

// The order of this lane's taskset: by priority desc, position asc.  False if a core has more than kTileOnCore tasks.
template <class Rows>
__device__ __forceinline__ bool tile_order(const Rows &rows, int n, bool best_effort, int &n_rt, int &n_gpu) {
  int pmax = (int)0x80000000;
#pragma unroll
  for (int k = 0; k < kTileCores; ++k) rows.on_core(k) = 0u;
  for (int i = 0; i < n; ++i) pmax = max(pmax, rows.priority(i));
  u32 seen = 0;
  n_rt = n, n_gpu = 0;
  for (int i = 0; i < n; ++i) {
    const int prio = rows.priority(i);
    const u32 word = rows.word(i);
    const u32 r = (u32)pmax - (u32)prio;
    if (r < (u32)n) rows.order(r) = (unsigned char)i, seen |= 1u << r;
    if (best_effort && prio <= 0) n_rt -= 1;
    n_gpu += tile_segments(word) != 0 ? 1 : 0;
    rows.on_core(word >> 28) |= 1u << i;
  }
  if (seen != (u32)((1ull << n) - 1ull)) {  // no dense numbering: count the tasks that come before
    for (int i = 0; i < n; ++i) {
      const int prio = rows.priority(i);
      int r = 0;
      for (int q = 0; q < n; ++q) {
        const int pq = rows.priority(q);
        r += (pq > prio || (pq == prio && q < i)) ? 1 : 0;
      }
      rows.order(r) = (unsigned char)i;
    }
  }
  int most = 0;
#pragma unroll
  for (int k = 0; k < kTileCores; ++k) most = max(most, __popc(rows.on_core(k)));
  return most <= kTileOnCore;
}

// The taskset of this lane, rank by rank (Eq. 1), all ranks narrow.  As in recurrence_narrow the quotients
// are exact and sums that are not exact exceed every deadline; here the sum over the GPU-using tasks runs
// over all of them with the weight of other cores, and what that counts too much for the same core is
// taken off again.  For a result R <= D that is at most twice what the same-core terms add (S <= W^c
// and ceil((R + J^g)/T) <= 2 ceil(R/T)), so every partial sum stays below 3 * 2^23/3 and is exact; if R > D, one
// of the sums is so far above D that no rounding hides it.
// Results of bounded tasks and of a miss go to out[position] (unless that is null); under GCAPS the sentinels of the tasks behind
// them too.  Returns GCAPS_SCHED_*, or -1 for a taskset that is left over.
template <int MODE, class Rows>
__device__ __forceinline__ int tile_walk(const Rows &rows, float ovh, bool literal, int n, int n_rt, int n_gpu, i64 *out) {
  constexpr bool kGcaps = MODE < 2;
  const f32x2 two23 = pack2(kTwo23, kTwo23), minus23 = pack2(-kTwo23, -kTwo23), zero = pack2(0.0f, 0.0f);
  float g_sum = 0.0f;  // of all W^g
  int n_list = 0;
  u32 done = 0, gpu_done = 0;  // positions bounded so far, GPU-using ones among them
  bool alive = n > 0;
  int how = GCAPS_SCHED_YES, ended = n_rt;
#pragma unroll 1
  for (int r = 0;; ++r) {
    const bool active = alive && r < n_rt;
    // entries of the longest list, and one
    const int longest = kGcaps ? __reduce_max_sync(kFull, active ? n_list + 1 : 0) : (int)__any_sync(kFull, active);
    if (longest == 0) break;
    const int i = active ? rows.order(r) : 0;
    const uint4 own = rows.own(i);
    const u32 front = active ? rows.on_core(own.x >> 28) & done : 0u;
    const float T = tile_period(own.x), D = __uint_as_float(own.y), A = __uint_as_float(own.z);
    const float Ge = fabsf(__uint_as_float(own.w));
    const bool gi = (int)own.w < 0;
    float S, base;
    if (kGcaps) {
      const float eta = (float)tile_segments(own.x);
      S = 2.0f * ovh * eta;
      base = A + Ge + S + (eta + 1.0f) * ovh;
    } else {
      S = rows.slot_time(i, own, active);
      base = A + Ge + (gi ? S * (float)(n_gpu - 1) : 0.0f);
    }
    const bool use_list = kGcaps && (MODE == 1 || gi);
    // ---- sweeps, with the interferers in registers ---------------------------------------------------
    const float nu = MODE == 3 ? (float)(n_gpu - __popc(front & gpu_done) + 1) : 0.0f;
    const int most_front = __reduce_max_sync(kFull, __popc(front));
    float R = base;
    bool go = active && !(R > D);
    // same-core entries: GCAPS an entry's two pairs (J, W) side by side, RR two entries side by side
    auto gcaps_entry = [&](int h, bool have, f32x2 &I, f32x2 &J, f32x2 &W) {
      float inv, jc, wc, jg, wg;
      rows.gcaps_core(ModeTag<MODE>(), h, ovh, inv, jc, wc, jg, wg);
      inv = have ? inv : 0.0f;
      I = pack2(inv, inv), J = pack2(jc, jg), W = pack2(have ? wc : 0.0f, have && use_list ? -wg : 0.0f);
    };
    auto rr_entry = [&](int h, bool have, float &inv, float &j, float &w) {
      float A_h, S_h;
      rows.rr_core(h, inv, j, A_h, S_h);
      inv = have ? inv : 0.0f, w = have ? (MODE == 3 ? fmaf(S_h, nu, A_h) : A_h) : 0.0f;
    };
    auto term = [&](f32x2 RR, f32x2 I, f32x2 J, f32x2 W, f32x2 acc) -> f32x2 {
      return fma2(add2(fma2_down(add2(RR, J), I, two23), minus23), W, acc);
    };
    // NC same-core entries and NL pairs of list entries in registers; MORE: there may be others
    auto run = [&](auto nc_tag, auto nl_tag, auto more_tag) {
      constexpr int NC = nc_tag, NL = kGcaps ? (int)nl_tag : 0, NX = kGcaps ? NC : NC / 2;
      constexpr bool MORE = more_tag;
      f32x2 CI[NX], CJ[NX], CW[NX], LI[NL + 1], LJ[NL + 1], LW[NL + 1];
      u32 rest = front;
      f32x2 once = zero;
#pragma unroll
      for (int q = 0; q < NX; ++q) {
        const bool have = rest != 0;
        const int h = have ? __ffs((int)rest) - 1 : i;
        rest &= rest - 1u;
        if (kGcaps) {
          gcaps_entry(h, have, CI[q], CJ[q], CW[q]);
        } else {
          const bool have1 = rest != 0;
          const int h1 = have1 ? __ffs((int)rest) - 1 : i;
          rest &= rest - 1u;
          float i0, j0, w0, i1, j1, w1;
          rr_entry(h, have, i0, j0, w0), rr_entry(h1, have1, i1, j1, w1);
          CI[q] = pack2(i0, i1), CJ[q] = pack2(j0, j1), CW[q] = pack2(w0, w1);
        }
        once = add2(once, CW[q]);
      }
#pragma unroll
      for (int q = 0; q < NL; ++q) rows.list(q, n_list, ovh, LI[q], LJ[q], LW[q]);
      if (base > 0.0f && D - base < (float)GCAPS_RTA_ITER_CAP) R = base + sum2(once) + (use_list ? g_sum : 0.0f);
      go = active && !(R > D);
      int left = kTileSweeps;
#pragma unroll 1
      while (__any_sync(kFull, go) && left > 0) {
        left -= 1;
        const f32x2 RR = pack2(R, R);
        f32x2 acc = zero, acc2 = zero, list = zero, list2 = zero;
#pragma unroll
        for (int q = 0; q < NX; ++q) {
          if (q & 1) acc2 = term(RR, CI[q], CJ[q], CW[q], acc2);
          else acc = term(RR, CI[q], CJ[q], CW[q], acc);
        }
#pragma unroll
        for (int q = 0; q < NL; ++q) {
          if (q & 1) list2 = term(RR, LI[q], LJ[q], LW[q], list2);
          else list = term(RR, LI[q], LJ[q], LW[q], list);
        }
        if (MORE) {
          u32 m = rest;
#pragma unroll 2
          for (int q = NC; q < most_front; ++q, m &= m - 1u) {
            const bool have = m != 0;
            const int h = have ? __ffs((int)m) - 1 : i;
            f32x2 I, J, W;
            if (kGcaps) {
              gcaps_entry(h, have, I, J, W);
            } else {
              float i0, j0, w0;
              rr_entry(h, have, i0, j0, w0);
              I = pack2(i0, 0.0f), J = pack2(j0, 0.0f), W = pack2(w0, 0.0f);
            }
            acc = term(RR, I, J, W, acc);
          }
          if (kGcaps) {
#pragma unroll 2
            for (int q = NL; 2 * q + 1 < longest; ++q) {
              f32x2 I, J, W;
              rows.list(q, n_list, ovh, I, J, W);
              list = term(RR, I, J, W, list);
            }
          }
        }
        float next = base + sum2(add2(acc, acc2));
        if (kGcaps) next += use_list ? sum2(add2(list, list2)) : 0.0f;
        const bool moved = go && next != R;
        R = moved ? next : R;
        go = moved && !(R > D);
      }
    };
    const int most_list = kGcaps ? longest >> 1 : 0;  // pairs
    if (most_front <= 2 && most_list <= 2) run(ModeTag<2>(), ModeTag<2>(), ModeTag<0>());
    else if (most_front <= 4 && most_list <= 4) run(ModeTag<4>(), ModeTag<4>(), ModeTag<0>());
    else if (most_front <= 6 && most_list <= 6) run(ModeTag<6>(), ModeTag<6>(), ModeTag<0>());
    else if (kGcaps && most_front <= 6 && most_list <= 9) run(ModeTag<6>(), ModeTag<9>(), ModeTag<0>());
    else run(ModeTag<6>(), ModeTag<6>(), ModeTag<1>());
    if (active) {
      if (R > D || go) {  // a miss; a taskset that has used up its sweeps is left over (their limit is part of the result)
        if (out) out[i] = GCAPS_WCRT_MISS;
        alive = false, ended = r + 1;
        how = R > D ? GCAPS_SCHED_NO : -1;
      } else {
        if (out) out[i] = (i64)(int)R;
        const float t = T - 0.5f, inv = __frcp_rn(T);
        if (kGcaps) {
          const float jg = (R - Ge) + t;
          rows.gcaps_publish(i, inv, MODE == 0 && gi ? (R - A) + t : t, MODE == 0 ? A + S : A + (gi ? Ge + S : 0.0f), jg, MODE == 0 ? S : Ge + S);
          if (gi) rows.append(n_list, i, inv, jg, Ge + S), n_list += 1, g_sum += Ge + S;
        } else {
          rows.rr_publish(i, inv, MODE == 2 && (gi || literal) ? (R - A) + t : t, A, S);
        }
        done |= 1u << i, gpu_done |= gi ? 1u << i : 0u;
      }
    }
  }
  if (kGcaps && out)
    for (int r = ended; r < n; ++r) out[rows.order(r)] = r < n_rt ? GCAPS_WCRT_SKIPPED : GCAPS_WCRT_BEST_EFFORT;
  return how;
}

// Whether the walks of a tile are worth while: not if three quarters of its tasksets have more tasks on a core than
// a walk is good for (60,000 tasksets of 16 tasks on one core 162 us, 110 in groups of lanes; 20 on two cores 134 and 144,
// 24 on two 171 and 162).  A few such tasksets in a tile (worst fit
// leaves one core with ten small tasks now and then) are no reason to start the launches behind, 25 us for any.
__device__ __forceinline__ bool tile_worth(bool taken, bool fits) {
  return 4 * __popc(__ballot_sync(kFull, taken && !fits)) < 3 * __popc(__ballot_sync(kFull, taken));
}

// Under round robin most tasks lie behind a miss: the results of the whole tile start as sentinels, which takes few
// stores where its tasksets follow one another in the batch.
__device__ __forceinline__ void tile_fill(i64 *out_wcrt, const TileLane &me, int lane) {
  const i64 end = __shfl_up_sync(kFull, me.a + me.n, 1);
  const u32 taken = __ballot_sync(kFull, me.n > 0), follows = __ballot_sync(kFull, me.n > 0 && end == me.a);
  const int last = 31 - __clz((int)taken);
  if (taken == 0) return;
  if ((taken & 1u) && (follows | 1u) == taken) {
    i64 *const out = out_wcrt + __shfl_sync(kFull, me.a, 0);
    const int all = (int)(__shfl_sync(kFull, me.a + me.n, last) - __shfl_sync(kFull, me.a, 0));
#pragma unroll 4
    for (int x = lane; x < all; x += 32) out[x] = GCAPS_WCRT_SKIPPED;
  } else {
#pragma unroll 1
    for (int c = 0; c <= last; ++c) {
      const int n = __shfl_sync(kFull, me.n, c);
      const i64 a = __shfl_sync(kFull, me.a, c);
      if (lane < n) out_wcrt[a + lane] = GCAPS_WCRT_SKIPPED;
    }
  }
  __syncwarp();
}

constexpr int kTileLeast = 4;  // rows
__host__ __device__ constexpr int tile_rows(int n) { return n < kTileLeast ? kTileLeast : n; }

// Whether the batch is one for tiles: of its sizes the host knows the mean only.  Every warp looks at the same 32 tasksets spread over
// the batch, and takes tiles if no more than four of them are larger than n or smaller than three quarters of it.  If more are,
// the tasksets are counted by size bins here, for the plan and the launches behind (plan_behind_tiles_kernel): in a mixture bins are
// the better way, whatever its mean.  100,000 tasksets, GCAPS / RR / all four analyses in tiles and in bins: 8 and 16 tasks
// alternating 170 / 139 / 428 and 129 / 109 / 355 us, 12 to 24 tasks 262 / 161 / 657 and 204 / 143 / 580, 8 and 40 tasks
// 1,089 / 316 / 1,941 and 404 / 149 / 991.
// look_into (where a warp has more than one tile): at the tasks of four of them too, a lane each.  If three are beyond what tiles take, or
// too crowded to be worth while (tile_worth), so is the batch.  100,000 tasksets of 8 tasks with long periods 181 / 130 / 529 us
// in tiles first and 111 / 94 / 327 straight in bins, 60,000 of 16 tasks on one core 123 / 108 / 330 and 98 / 93 / 289.
// A function of its own: inlined, the registers that it holds for a moment made the walks spill (25 pairs 561 -> 587 us with eight
// tasksets looked into, 574 with four).
constexpr int kLookedInto = 4;
__device__ __noinline__ bool tile_batch(const i64 *task_off, const i64 *period, const i64 *core, i64 n_tasksets, i64 n_tasks, i64 task_base,
                                        PlanHeader *hdr, int n, bool look_into) {
  const int lane = threadIdx.x & 31;
  const i64 stride = n_tasksets / 32, t = lane * stride + (i64)((lane * 2654435761u) >> 8) % stride;  // (at odd distances: kinds may alternate)
  const i64 first = task_off[t] - task_base, end = task_off[t + 1] - task_base;
  const int other_sizes = __popc(__ballot_sync(kFull, end - first > n || 4 * (end - first) < 3 * n));
  u64 T[kLookedInto], c[kLookedInto];
#pragma unroll
  for (int k = 0; k < kLookedInto; ++k) {
    const i64 a = __shfl_sync(kFull, first, 32 / kLookedInto * k), b = __shfl_sync(kFull, end, 32 / kLookedInto * k);
    T[k] = 0, c[k] = 0x100 + lane;  // (no task: a core of its own)
    if (look_into && a >= 0 && b <= n_tasks && b - a <= n && lane < b - a) T[k] = (u64)period[a + lane], c[k] = (u64)core[a + lane];
  }
  int in_vain = 0;
#pragma unroll
  for (int k = 0; k < kLookedInto; ++k) {
    const bool crowded = __popc(__match_any_sync(kFull, (u32)c[k])) > kTileOnCore;
    in_vain += __any_sync(kFull, T[k] >= kNarrowLimit || (T[k] > 0 && c[k] >= kTileCores) || crowded) ? 1 : 0;
  }
  if (other_sizes <= 4 && 4 * in_vain < 3 * kLookedInto) {
    if (blockIdx.x == 0 && lane == 0) hdr->in_tiles = 1;
    return true;
  }
  u32 counts[kNumBins];
#pragma unroll
  for (int k = 0; k < kNumBins; ++k) counts[k] = 0;
#pragma unroll 4
  for (i64 t0 = (i64)blockIdx.x * 32; t0 < n_tasksets; t0 += (i64)gridDim.x * 32) {
    const int bin = t0 + lane < n_tasksets ? size_bin(task_off[t0 + lane + 1] - task_off[t0 + lane]) : kNumBins;
#pragma unroll
    for (int k = 0; k < kNumBins; ++k) counts[k] += __popc(__ballot_sync(kFull, bin == k));
  }
#pragma unroll
  for (int k = 0; k < kNumBins; ++k)
    if (lane == k && counts[k] > 0) atomicAdd(&hdr->bin_count[k], counts[k]);
  return false;
}

// The tasksets of a batch of n tasks each in its order, a tile per warp at a time.  `rows`: where the tasks are kept, room for
// tile_rows(n) positions of Rows::kSets tasksets.  walk(tile lane) analyses the tile; false in the lane of a taskset that is left over.
// What tiles do not take is listed in the workspace, for the launches behind this one: tasksets that fit the size bin of
// n tasks as that bin, from the front on, all others as bin kRestLarge from the end on.
template <bool SLICES, class Rows, class Walk>
__device__ __forceinline__ void run_tiles(const KParams &p, int n, const Rows &rows, Walk walk) {
  const unsigned int count = (unsigned int)p.n_tasksets;
  const int lane = threadIdx.x & 31, n_rows = tile_rows(n), small_bin = (n - 1) / 8;
  // columns per tile: as many as give every warp the same number of tiles
  const unsigned int rounds = (count + Rows::kSets * gridDim.x - 1) / (Rows::kSets * gridDim.x);
  unsigned int chunk = (count + rounds * gridDim.x - 1) / (rounds * gridDim.x);
  chunk = chunk < 4 ? 4 : chunk;

  auto pull = [&]() -> unsigned int { return lane == 0 ? atomicAdd(&p.hdr->next[kNextTile], chunk) : 0u; };
  auto look_up = [&](unsigned int first, TileLane &x, i64 &b) {
    const bool mine = (unsigned int)lane < chunk && first < count && first + lane < count;
    x.t = mine ? first + lane : kNoTaskset;
    x.a = x.c = x.g = 0, x.n = x.size = 0, x.nc = x.ng = 0, x.declined = false, b = 0;
    if (mine) x.a = p.task_off[x.t] - p.task_base, b = p.task_off[(i64)x.t + 1] - p.task_base;
  };
  auto settle = [&](TileLane &x, i64 b) {
    if (x.t == kNoTaskset) return;
    x.declined = true;
    if (x.a < 0 || b <= x.a || b > p.n_tasks || b - x.a > GCAPS_RTA_MAX_TASKS) return;
    x.size = (int)(b - x.a);
    if (x.size <= n_rows) {
      x.c = p.cseg_off[x.a] - p.cseg_base, x.g = p.gseg_off[x.a] - p.gseg_base;
      const i64 c_hi = p.cseg_off[b] - p.cseg_base, g_hi = p.gseg_off[b] - p.gseg_base;
      if (x.c >= 0 && c_hi >= x.c && c_hi <= p.n_csegs && x.g >= 0 && g_hi >= x.g && g_hi <= p.n_gsegs &&
          c_hi - x.c < 64 * 32 && g_hi - x.g < rows.most_gsegs())
        x.n = x.size, x.nc = (u32)(c_hi - x.c), x.ng = (u32)(g_hi - x.g), x.declined = false;
    }
  };
  // A tile's loads come out of L2: while the tile in front of it is worked on, each lane asks for the lines
  // of its taskset.
  auto ask_for = [&](const i64 *from, i64 first, i64 to) {
    for (i64 e = first; e < to; e = (e | 15) + 1) prefetch_l2(from + e);
  };
  auto list = [&](bool wanted, u32 t, int bin) {
    const u32 bits = __ballot_sync(kFull, wanted);
    if (bits == 0) return;
    unsigned int at = 0;
    if (lane == 0) at = atomicAdd(&p.hdr->bin_count[bin], (unsigned int)__popc(bits));
    at = __shfl_sync(kFull, at, 0) + __popc(bits & ((1u << lane) - 1u));
    if (wanted) p.perm[bin == kRestLarge ? count - 1u - at : at] = t;
  };
  unsigned int first = __shfl_sync(kFull, pull(), 0), second = __shfl_sync(kFull, pull(), 0);
  TileLane me, coming;
  i64 b;
  look_up(first, me, b);
  if (!tile_batch(p.task_off, p.period, p.core, p.n_tasksets, p.n_tasks, p.task_base, p.hdr, n, rounds > 1)) return;
  settle(me, b);
  TilePatience patience = {0};
#pragma unroll 1
  while (first < count) {
    const bool looks = patience.looks();
    if (!looks && me.n > 0) me.declined = true, me.n = 0;
    const unsigned int asked = pull();
    const int columns = count - first < chunk ? (int)(count - first) : (int)chunk;
    look_up(second, coming, b);
#pragma unroll 1
    for (int c0 = 0; looks && c0 < columns; c0 += 32 / kTileGroup) {
      if (n_rows <= 8) tile_stage<1, SLICES>(p, rows, me, c0, lane);
      else if (n_rows <= 16) tile_stage<2, SLICES>(p, rows, me, c0, lane);
      else tile_stage<3, SLICES>(p, rows, me, c0, lane);
      // (none of the first ones: nor the others of this tile, for an eighth of its stage)
      if (c0 == 0 && columns >= 4 && (__ballot_sync(kFull, me.declined) & 0xfu) == 0xfu) {
        if (me.n > 0) me.declined = true, me.n = 0;
        break;
      }
    }
    __syncwarp();
    const unsigned int third = __shfl_sync(kFull, asked, 0);
    settle(coming, b);
    if (coming.n > 0 && patience.unseen <= 1) {
      const i64 to = coming.a + coming.n;
      ask_for(p.cseg_off, coming.a, to), ask_for(p.gseg_off, coming.a, to);
      ask_for(p.period, coming.a, to), ask_for(p.deadline, coming.a, to), ask_for(p.priority, coming.a, to), ask_for(p.core, coming.a, to);
      ask_for(p.cseg_wcet, coming.c, coming.c + coming.nc);
      ask_for(p.gseg_misc, coming.g, coming.g + coming.ng), ask_for(p.gseg_exec, coming.g, coming.g + coming.ng);
    }
    __syncwarp();
    if (!walk(me) && me.n > 0) me.declined = true;
    const bool small = me.size >= 1 && me.size <= 8 * (small_bin + 1);
    list(me.declined && small, me.t, small_bin);
    list(me.declined && !small, me.t, kRestLarge);
    patience.done(__popc(__ballot_sync(kFull, me.declined && me.n > 0)), columns);
    __syncwarp();
    me = coming;
    first = second, second = third;
  }
}

}  // namespace
#endif  // GCAPS_RTA_TILE_CUH_
