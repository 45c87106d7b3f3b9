// rta_recurrence.cuh -- the recurrence of Eq. 1 for the tasks of one taskset in rank order, once
// every task's values lie in shared memory in the row of its rank.  Internal; included by
// rta_device.cuh.
//
// recurrence_narrow works in single precision with exact integer results and takes the ranks in
// front of the first one whose period reaches kNarrowLimit (2.8 s); recurrence_wide continues from
// there in 32-bit integers.
//
// Why single precision.  The recurrence is bound by instruction issue and by the multiply pipe.
// With every time below 2^23 / 3 the dividend x = R + J + T_h - 1/2 is a multiple of 1/2 below
// 2^23, so it is a float, and floor(x / T_h) = ceil((R + J) / T_h) is one multiply-add rounded
// towards minus infinity: x * inv + 2^23 with inv = 1/T_h rounded to nearest.  Its error
// x * |inv - 1/T_h| <= (x / T_h) * 2^-24 < (1/2) / T_h, and x / T_h (an odd multiple of 1/2 over
// T_h) is at least (1/2) / T_h away from every integer, so the quotient is exact.  Quotient times
// weight is summed in a float too: exact below 2^24, and every rounding is monotone, so a sum
// that is not exact still exceeds every deadline.  Two pairs (J, W) go through one packed
// instruction (f32x2).  Per pair that is 2 issue slots; the integer form (multiply-high, shift,
// 64-bit multiply-add) takes 6, four of them on the half-rate multiply pipe.
#ifndef GCAPS_RTA_RECURRENCE_CUH_
#define GCAPS_RTA_RECURRENCE_CUH_

#include <cuda_runtime.h>
#include <stdint.h>

#include "rta_common.cuh"

namespace {

using namespace gcaps_detail;

constexpr u32 kNarrowLimit = 2796200u;  // periods below this: x < 3 * kNarrowLimit < 2^23
constexpr u32 kOne23 = 0x4B000000u;     // the bits of 2^23; 2^23 + k for 0 <= k < 2^23 is kOne23 + k
constexpr float kTwo23 = 8388608.0f;
constexpr u32 kRowGpu = 0x80000000u;

template <int LPT, int SLOTS>
struct FastLayout {
  static constexpr int MAXN = LPT * SLOTS;
  static constexpr int kStep = 4 * LPT;  // elements one prefix step of the group covers
  // a prefix array takes slices of up to CAP-1 elements (a taskset with more goes through the 64-bit
  // path) and is written kStep words at a time.  Small tasksets vary more: 8 per task (200,000 tasksets
  // of `divergence` under GCAPS 480 -> 455 us against 6 per task)
  static constexpr int CAP = ((LPT == 32 ? 6 : 8) * MAXN + kStep - 1) / kStep * kStep;
  static constexpr int kInfo = 0;  // row A by rank
  static constexpr int kQ0 = 4 * MAXN + 4;
  static constexpr int kQ1 = kQ0 + CAP + 4;
  static constexpr int kFastWords = kQ1 + CAP;
  static constexpr int kExactWords = (17 * MAXN + 3) / 4 * 4;  // the exact path: 66 B per task
  static constexpr int kMost = kFastWords > kExactWords ? kFastWords : kExactWords;
  // the groups of a warp read the rows of the same rank together: their areas start on different
  // banks
  static constexpr int kWords = LPT == 32 ? kMost : (kMost + 31) / 32 * 32 + LPT;
  static_assert(kWords % 4 == 0 && CAP % kStep == 0 && 4 * MAXN <= CAP, "16-byte aligned rows");
};

// What the rows of a rank hold.  They are written as integers; recurrence_narrow turns a block of
// LPT ranks into single precision when it reaches the block (a taskset that misses early never
// pays for the rest), which is what stands in brackets:
//   row A  .x deadline [bits of 2^23 + D]   .y core   .z [1/T_h]
//   row B  .x T_h [float]   .y C+G^m [float]   .z G^e [float] with bit 31 = uses the GPU   .w S =
//          2*eps*eta (GCAPS) or (L+theta)*slices (RR), an integer throughout; in a sweep .w is R
//   one analysis: base[r] [bits of 2^23 + base, clamped], R[r]
//   sweep: second row  .x GPU segment range | eta << 22   .y slices of Eq. 3 for the timeslice
template <int LPT, int SLOTS, bool SWEEP>
struct Rows {
  typedef FastLayout<LPT, SLOTS> Lay;
  u32 *buf;
  __device__ __forceinline__ uint4 &a(int r) const { return reinterpret_cast<uint4 *>(buf + Lay::kInfo)[r]; }
  __device__ __forceinline__ uint4 &b(int r) const { return reinterpret_cast<uint4 *>(buf + Lay::kQ0)[r]; }
  __device__ __forceinline__ uint2 &second(int r) const {
    return reinterpret_cast<uint2 *>(buf + Lay::kQ0 + 4 * Lay::MAXN)[r];
  }
  __device__ __forceinline__ u32 &base(int r) const { return buf[Lay::kQ0 + 4 * Lay::MAXN + r]; }
  __device__ __forceinline__ u32 &R(int r) const {
    return SWEEP ? buf[Lay::kQ0 + 4 * r + 3] : buf[Lay::kQ0 + 5 * Lay::MAXN + r];
  }
};

// The constants of one (timeslice, overhead) pair.
struct PairConsts {
  u32 ovh;        // below 2^20 on the 32-bit path
  u64 slot_cost;  // L + theta
};

// S and base of a task from integers (clamped as on the 32-bit path: a clamped value exceeds every
// deadline).  GCAPS: S = 2*eps*eta, base = C_i + G*_i + B^C_i; RR: S = (L+theta)*slices, Lemma 1.
template <bool GCAPS>
__device__ __forceinline__ void own_cost(const PairConsts &pc, u32 A, u32 Ge, u32 eta, u32 slices, int n_gpu,
                                         u32 &S, u32 &base) {
  if (GCAPS) {
    S = 2 * pc.ovh * eta;                        // eta < 64: below 2^27
    base = A + Ge + S + (eta + 1) * pc.ovh;      // below 2^29
  } else {
    u64 B = slices == 0 ? 0 : (pc.slot_cost >= kFastClamp ? kFastClamp : pc.slot_cost * (u64)slices);
    if (B > kFastClamp) B = kFastClamp;
    S = (u32)B;
    const u64 b64 = (u64)A + Ge + (eta > 0 ? B * (u64)(n_gpu - 1) : 0);
    base = b64 > (u64)(2 * kFastClamp) ? 2 * kFastClamp : (u32)b64;
  }
  base = base > 2 * kFastClamp ? 2 * kFastClamp : base;
}

// ---- packed single precision ------------------------------------------------------------------
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float sum2(f32x2 v) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
  return lo + hi;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 fma2_down(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

template <int LPT>
__device__ __forceinline__ bool group_all(bool x, unsigned int gmask) {
  if constexpr (LPT == 32) return __all_sync(kFull, x);
  return (__ballot_sync(kFull, x) & gmask) == gmask;
}

// How a recurrence ended: ranks below n_done converged (their R is in the rows); verdict 0, or what
// rank n_done gets.
struct Outcome {
  int n_done, verdict;
};

// Ranks 0 .. n_f-1 of a group's taskset (n_f = 0: nothing to do), all rows narrow.  Called by the
// whole warp: its groups walk through the ranks side by side, and at every rank they sweep until
// the last of them has converged (a converged group repeats its fixed point), so nothing diverges
// and every collective is one instruction for the whole warp.  A lane keeps, in registers, what
// the tasks of rank lane, lane + LPT, ... contribute as interferers; a task not yet bounded has
// inv = 0 there, which makes its quotient 0.  The loop over a block of LPT ranks is compiled once
// per number of slots in use.
//
// The first iterate.  For base_i > 0 every ceiling is at least 1, so base_i + sum of all W_h is not
// above the least fixed point; it costs a sweep without its divisions, so the iteration starts
// there: 318 -> 245 sweeps per taskset where all 80 tasks converge.  Only where D_i - base_i <
// GCAPS_RTA_ITER_CAP: a longer climb from base_i could run into the sweep limit, which is part of
// the result.
// `blocks_made`: blocks of ranks already in single precision (kept across the analyses of a sweep).
template <int LPT, int SLOTS, int MODE, bool SWEEP, class RowsT>
__device__ __forceinline__ Outcome recurrence_narrow(const RowsT rows, int n_f, int n_gpu,
                                                     const PairConsts &pc, bool literal, int lane,
                                                     unsigned int gmask, int &blocks_made) {
  constexpr bool kGcaps = MODE < 2;
  Outcome out;
  out.n_done = n_f, out.verdict = 0;
  // by slot: 1/T, the two dividends' constants, the weights, the core
  float inv[SLOTS], Ja[SLOTS], Jb[SLOTS], Wa[SLOTS], Wb[SLOTS], Wc[SLOTS];
  f32x2 inv2[SLOTS], J2s[SLOTS];  // MODE 0: (1/T, 1/T) and (J^c, J^g), as the sweeps take them
  u32 core[SLOTS];
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    inv[s] = Ja[s] = Jb[s] = Wa[s] = Wb[s] = Wc[s] = 0.0f, core[s] = 0xffffffffu;
    inv2[s] = J2s[s] = pack2(0.0f, 0.0f);
  }
  const f32x2 two23 = pack2(kTwo23, kTwo23), minus23 = pack2(-kTwo23, -kTwo23);
  const float ovh_f = (float)pc.ovh;
  const float slot_f = pc.slot_cost >= kFastClamp ? (float)kFastClamp : (float)(u32)pc.slot_cost;
  bool alive = n_f > 0;

#pragma unroll
  for (int blk = 0; blk < SLOTS; ++blk) {
    if (LPT == 32 ? n_f <= LPT * blk : !__any_sync(kFull, alive && n_f > LPT * blk)) return out;
    if (!SWEEP || blocks_made <= blk) {
      blocks_made = blk + 1;
      const int r = LPT * blk + lane;
      if (r < n_f) {
        uint4 fa = rows.a(r), fb = rows.b(r);
        const float T = (float)fb.x;
        fa.x += kOne23, fa.z = __float_as_uint(__frcp_rn(T));
        fb.x = __float_as_uint(T), fb.y = __float_as_uint((float)fb.y);
        fb.z = __float_as_uint((float)(fb.z & ~kRowGpu)) | (fb.z & kRowGpu);
        rows.a(r) = fa, rows.b(r) = fb;
        if (!SWEEP) {
          const u32 base = rows.base(r);
          rows.base(r) = kOne23 + (base < 0x7fffffu ? base : 0x7fffffu);
        }
      }
      __syncwarp();
    }
#pragma unroll 1
    for (int pos = LPT * blk; pos < LPT * (blk + 1); ++pos) {
      const bool active = alive && pos < n_f;
      if constexpr (LPT == 32) {
        if (!active) return out;
      } else {
        if (!__any_sync(kFull, active)) return out;
      }
      // ---- the task under analysis -------------------------------------------------------------
      const uint4 fa = rows.a(pos), fb = rows.b(pos);
      const float Db = __uint_as_float(fa.x);
      const u32 core_i = fa.y;
      const float T = __uint_as_float(fb.x), A = __uint_as_float(fb.y), Ge = fabsf(__uint_as_float(fb.z));
      const bool gi = (int)fb.z < 0;
      float S, base_b;  // base_b = 2^23 + base
      if constexpr (SWEEP) {
        const uint2 g = rows.second(pos);
        const float eta = (float)(g.x >> 22);
        float base;
        if (kGcaps) {
          S = 2.0f * ovh_f * eta;
          base = A + Ge + S + (eta + 1.0f) * ovh_f;
        } else {
          S = g.y == 0 ? 0.0f : fminf(slot_f * (float)g.y, (float)kFastClamp);
          base = A + Ge + (gi ? S * (float)(n_gpu - 1) : 0.0f);
        }
        base_b = fminf(base, kTwo23 - 1.0f) + kTwo23;
      } else {
        S = (float)fb.w;
        base_b = __uint_as_float(rows.base(pos));
      }
      float nu = 0.0f;
      if (MODE == 3) {  // Lemma 4: N_g - |{h in hpp(i): GPU-using}| + 1
        int c = 0;
#pragma unroll
        for (int s = 0; s <= blk; ++s)
          c += __popc(__ballot_sync(kFull, inv[s] != 0.0f && core[s] == core_i && Wc[s] != 0.0f) & gmask);
        nu = (float)(n_gpu - c + 1);
      }
      // ---- the (J, W) pairs of this task's interferers; W = 0 where a pair does not apply ---------
      constexpr int kPairs = SLOTS + 1;  // packed pairs: MODE 0 two pairs of one slot, else two slots
      f32x2 I2[kPairs], J2[kPairs], W2[kPairs];
      if (MODE == 0) {
#pragma unroll
        for (int s = 0; s <= blk; ++s) {
          // Lemma 15, jitter J^c; Lemma 13 (same core | other cores), jitter J^g.  Only the weights depend on the task
          // under analysis
          const bool same = core[s] == core_i;
          const float wg = same ? Wc[s] : Wb[s];
          I2[s] = inv2[s], J2[s] = J2s[s], W2[s] = pack2(same ? Wa[s] : 0.0f, gi ? wg : 0.0f);
        }
      } else {
        float j[SLOTS + 1], w[SLOTS + 1], d[SLOTS + 1];
        const bool all_of_it = gi || !literal;
#pragma unroll
        for (int s = 0; s <= blk; ++s) {
          const bool same = core[s] == core_i;
          d[s] = inv[s];
          if (MODE == 1) {
            w[s] = same ? (all_of_it ? Wc[s] : Wa[s]) : Wb[s];  // Lemmas 12+10 / 10, 11
            j[s] = same ? Ja[s] : Jb[s];
          } else if (MODE == 2) {
            w[s] = same ? Wa[s] : 0.0f;                         // Lemma 7
            j[s] = Ja[s];
          } else {
            w[s] = same ? fmaf(Wb[s], nu, Wa[s]) : 0.0f;        // Lemmas 5 and 4
            j[s] = Ja[s];
          }
        }
        d[blk + 1] = j[blk + 1] = w[blk + 1] = 0.0f;
#pragma unroll
        for (int k = 0; k <= blk / 2; ++k)
          I2[k] = pack2(d[2 * k], d[2 * k + 1]), J2[k] = pack2(j[2 * k], j[2 * k + 1]), W2[k] = pack2(w[2 * k], w[2 * k + 1]);
      }
      constexpr bool kOnePair = MODE == 0;
      const int n_pairs = kOnePair ? blk + 1 : blk / 2 + 1;
      // base + the group's sum, as 2^23 + value.  A warp per taskset: the lanes' sums (started at
      // 2^23, so that their bits count) are added as integers; smaller groups add floats.
      const u32 base_bits = __float_as_uint(base_b) - 32u * kOne23;
      const f32x2 acc0 = LPT == 32 ? pack2(kTwo23, 0.0f) : pack2(0.0f, 0.0f);
      auto total = [&](f32x2 acc) -> float {
        float f = sum2(acc);
        if constexpr (LPT == 32) {
          f = fminf(f, kTwo23 + 4194304.0f);  // 2^22 exceeds every narrow deadline
          return __uint_as_float(__reduce_add_sync(kFull, __float_as_uint(f)) + base_bits);
        } else {
#pragma unroll
          for (int d = 1; d < LPT; d <<= 1) f += __shfl_xor_sync(kFull, f, d);
          return base_b + f;
        }
      };
      auto sweep = [&](float R) -> float {
        const f32x2 RR = pack2(R, R);
        f32x2 acc = acc0;
#pragma unroll
        for (int k = 0; k < n_pairs; ++k) {
          const f32x2 q = fma2_down(add2(RR, J2[k]), I2[k], two23);
          acc = fma2(add2(q, minus23), W2[k], acc);
        }
        return total(acc);
      };
      f32x2 acc = acc0;
#pragma unroll
      for (int k = 0; k < n_pairs; ++k) acc = add2(acc, W2[k]);
      const float all_once = total(acc);
      float R = (Db - base_b < (float)GCAPS_RTA_ITER_CAP && base_b > kTwo23) ? all_once : base_b;
      // ---- sweeps ---------------------------------------------------------------------------------
      int left = (int)GCAPS_RTA_ITER_CAP, verdict = 0;
      if constexpr (LPT == 32) {
        if (R > Db) {
          verdict = GCAPS_WCRT_MISS;
        } else {
          for (;;) {
            if (left == 0) {
              verdict = GCAPS_WCRT_ITER_LIMIT;
              break;
            }
            left -= 1;
            const float next = sweep(R);
            if (next == R) break;
            R = next;
            if (R > Db) {
              verdict = GCAPS_WCRT_MISS;
              break;
            }
          }
        }
        if (verdict != 0) {
          out.n_done = pos, out.verdict = verdict;
          return out;
        }
      } else {
        bool go = active && !(R > Db);
#pragma unroll 1
        while (__any_sync(kFull, go) && left > 0) {
          left -= 1;
          const float next = sweep(R);
          const bool moved = go && next != R;
          R = moved ? next : R;
          go = moved && !(R > Db);
        }
        if (active && (go || R > Db)) {
          out.n_done = pos, out.verdict = R > Db ? GCAPS_WCRT_MISS : GCAPS_WCRT_ITER_LIMIT;
          alive = false;
        }
      }
      // ---- publish: R_i, and what the owner's lane holds of this task from now on -----------------
      // (the jitters J^c = R - (C+G^m), J^g = R - G^e enter as J + T - 1/2 - 2^23; a CPU-only task
      // has no J^c unless the printed form of Lemma 7 is asked for)
      if (active && alive) {
        if (lane == 0) rows.R(pos) = __float_as_uint(R) - kOne23;
        if (lane == pos - LPT * blk) {
          const float t = (T - 0.5f) - kTwo23, Rp = R - kTwo23;
          inv[blk] = __uint_as_float(fa.z), core[blk] = core_i;
          if (MODE == 0) {
            inv2[blk] = pack2(inv[blk], inv[blk]), J2s[blk] = pack2(gi ? (Rp - A) + t : t, (Rp - Ge) + t);
            Wa[blk] = A + S;      // Lemma 15: C_h, or C_h + G^{m*}_h (S = 0 for a CPU-only task)
            Wb[blk] = Ge + S;     // Lemma 13, other cores: G^{e*}_h
            Wc[blk] = Ge;
          } else if (MODE == 1) {
            Ja[blk] = t, Jb[blk] = (Rp - Ge) + t;
            Wa[blk] = A;          // Lemma 12
            Wb[blk] = Ge + S;     // Lemmas 10, 11: G^{e*}_h
            Wc[blk] = A + (Ge + S);
          } else {
            Ja[blk] = (MODE == 2 && (gi || literal)) ? (Rp - A) + t : t;
            Wa[blk] = A;          // Lemmas 5, 7
            Wb[blk] = S;          // Lemma 4: (L+theta) * slices
            Wc[blk] = gi ? 1.0f : 0.0f;
          }
        }
      }
    }
  }
  return out;
}

// The ranks from `start` on in 32-bit integers (every time below 2^26): the continuation behind the
// first period of kNarrowLimit or more.  Rare (a taskset must have converged up to there), hence
// not inlined.  Called by the lanes of one group.
template <int LPT, int SLOTS, int MODE, bool SWEEP>
__device__ __noinline__ Outcome recurrence_wide(u32 *buf, int n, int n_rt, int start, int n_gpu, PairConsts pc,
                                                bool literal, int lane, unsigned int gmask) {
  constexpr bool kGcaps = MODE < 2;
  const Rows<LPT, SLOTS, SWEEP> rows{buf};
  struct Task {
    u32 D, core, T, A, Ge, S, base;
    bool gpu;
  };
  auto load = [&](int r) -> Task {
    Task k;
    const uint4 fa = rows.a(r), fb = rows.b(r);
    k.core = fa.y, k.gpu = (fb.z & kRowGpu) != 0;
    const u32 ge = fb.z & ~kRowGpu;
    if (r >= start) {
      k.D = fa.x, k.T = fb.x, k.A = fb.y, k.Ge = ge;
    } else {  // (in single precision by now)
      k.D = fa.x - kOne23, k.T = (u32)__uint_as_float(fb.x), k.A = (u32)__uint_as_float(fb.y);
      k.Ge = (u32)__uint_as_float(ge);
    }
    if constexpr (SWEEP) {
      const uint2 g = rows.second(r);
      own_cost<kGcaps>(pc, k.A, k.Ge, g.x >> 22, g.y, n_gpu, k.S, k.base);
    } else {
      k.S = fb.w;
      k.base = rows.base(r);  // (only read from `start` on)
    }
    return k;
  };
  u32 Tm1[SLOTS], Ar[SLOTS], Ger[SLOTS], core[SLOTS], Wa[SLOTS], Wb[SLOTS], magic[SLOTS], shift[SLOTS];
  u32 Jc[SLOTS], Jg[SLOTS];  // jitters with T_h - 1 folded in (ceiling)
  bool gpu[SLOTS];
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    const int r = lane + LPT * s;
    Task k;
    k.D = 0, k.core = 0xffffffffu, k.T = 2, k.A = k.Ge = k.S = k.base = 0, k.gpu = false;
    if (r < n) k = load(r);
    Tm1[s] = k.T - 1, Ar[s] = k.A, Ger[s] = k.Ge, core[s] = k.core, gpu[s] = k.gpu;
    make_reciprocal(k.T, magic[s], shift[s]);
    Wa[s] = k.A + ((MODE == 0 && k.gpu) ? k.S : 0u);
    Wb[s] = k.gpu ? (MODE < 2 ? k.Ge + k.S : k.S) : 0u;
    Jc[s] = Jg[s] = Tm1[s];
    if (r < start) {
      const u32 R = rows.R(r);
      if (MODE == 0 ? k.gpu : (MODE == 2 ? (k.gpu || literal) : false)) Jc[s] = R - k.A + Tm1[s];
      Jg[s] = R - k.Ge + Tm1[s];
    }
  }
  Outcome out;
  out.n_done = n_rt, out.verdict = 0;
  for (int pos = start; pos < n_rt; ++pos) {
    const Task me = load(pos);
    u32 nu = 0;
    if (MODE == 3) {  // Lemma 4: N_g - |{h in hpp(i): GPU-using}| + 1
      int c = 0;
#pragma unroll
      for (int s = 0; s < SLOTS; ++s)
        c += __popc(__ballot_sync(gmask, lane + LPT * s < pos && core[s] == me.core && gpu[s]));
      nu = (u32)(n_gpu - c + 1);
    }
    u32 J1[SLOTS], W1[SLOTS], W2[SLOTS];
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      const bool act = lane + LPT * s < pos, same = core[s] == me.core;
      u32 w1, w2 = 0, j1;
      if (MODE == 0) {
        w1 = same ? Wa[s] : (me.gpu ? Wb[s] : 0u);
        j1 = same ? Jc[s] : Jg[s];
        w2 = (same && me.gpu && gpu[s]) ? Ger[s] : 0u;
      } else if (MODE == 1) {
        w1 = same ? Wa[s] + ((me.gpu || !literal) ? Wb[s] : 0u) : Wb[s];
        j1 = same ? Tm1[s] : Jg[s];
      } else if (MODE == 2) {
        w1 = same ? Wa[s] : 0u;
        j1 = Jc[s];
      } else {
        const u64 w = (u64)Wa[s] + (u64)Wb[s] * nu;
        w1 = same ? (w > kFastClamp ? kFastClamp : (u32)w) : 0u;
        j1 = Tm1[s];
      }
      J1[s] = j1, W1[s] = act ? w1 : 0u, W2[s] = act ? w2 : 0u;
    }
    u32 R = me.base;
    int v = 0;
    for (int sweeps = 0;; ++sweeps) {
      if (R > me.D) {
        v = GCAPS_WCRT_MISS;
        break;
      }
      if (sweeps >= (int)GCAPS_RTA_ITER_CAP) {
        v = GCAPS_WCRT_ITER_LIMIT;
        break;
      }
      u64 acc = 0;
#pragma unroll
      for (int s = 0; s < SLOTS; ++s) {
        acc += (u64)(__umulhi(R + J1[s], magic[s]) >> shift[s]) * W1[s];
        if (MODE == 0) acc += (u64)(__umulhi(R + Jg[s], magic[s]) >> shift[s]) * W2[s];
      }
      const u32 part = acc > (u64)kFastClamp ? kFastClamp : (u32)acc;
      const u32 next = me.base + __reduce_add_sync(gmask, part);
      if (next == R) break;
      R = next;
    }
    if (v != 0) {
      out.n_done = pos, out.verdict = v;
      break;
    }
    if (lane == 0) rows.R(pos) = R;
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      if (lane + LPT * s == pos) {
        if (MODE == 0 ? gpu[s] : (MODE == 2 ? (gpu[s] || literal) : false)) Jc[s] = R - Ar[s] + Tm1[s];
        Jg[s] = R - Ger[s] + Tm1[s];
      }
    }
  }
  __syncwarp(gmask);
  return out;
}

}  // namespace
#endif  // GCAPS_RTA_RECURRENCE_CUH_
