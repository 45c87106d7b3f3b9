// rta_tile_kept.cuh -- several analyses per taskset of tasksets of up to 24 tasks: a tile is staged and ordered once,
// then every taskset has Q lanes, each of which takes it through the recurrence under another analysis or (timeslice,
// overhead) pair.  Internal.
#ifndef GCAPS_RTA_TILE_KEPT_CUH_
#define GCAPS_RTA_TILE_KEPT_CUH_

#include "rta_tile.cuh"

namespace {

constexpr int kKindGcaps = 1, kKindRr = 2;
constexpr int kKeptFew = 2;  // walks of a policy up to which a taskset has two lanes; with more it has four

// Shared memory of one warp's tile of 32/Q tasksets.  A row holds what belongs to the task of a position, for every column,
//   own  T and more, D, A = C+G^m, G^e with the sign bit = uses the GPU
//   inv  1/T
// and what a walk knows of it, for every lane,
//   x    (priority, by column, before the walks) J^c (GCAPS), J (RR)
//   y    J^g (GCAPS), slices of Eq. 3 (RR)
// Behind the rows, by column: positions by core (bits) and by rank; under GCAPS the positions of the GPU-using tasks in
// rank order; under RR the pure GPU parts' times and, by position, where a task's start.
template <int KINDS, int Q>
struct KeptRows {
  static constexpr int kSets = 32 / Q;
  static constexpr int kStride = kSets + 1;  // the stage writes with lanes at different rows of one column
  // an odd number of 16-byte units: rows of a column start on different banks
  static constexpr int kRow = 16 * ((20 * kStride + 256 + 15) / 16 | 1);
  static constexpr int kInv = 16 * kStride, kX = (20 * kStride + 15) / 16 * 16, kY = kX + 128;
  static_assert(kY + 128 <= kRow, "a row holds both lane planes");
  unsigned char *mem, *ord, *lst, *goff;
  u32 *cores, *segs;
  int seg_room;  // words per column
  int lane, col, sub;

  static __host__ __device__ constexpr int bytes(int rows, int segments) {
    return rows * kRow + kTileCores * kSets * 4 + ((KINDS & kKindRr) ? kSets * (segments | 1) * 4 : 0) + rows * kSets +
           ((KINDS & kKindGcaps) ? rows * kSets : 0) + ((KINDS & kKindRr) ? rows * kSets : 0);
  }
  __device__ __forceinline__ KeptRows(unsigned char *at, int rows, int segments) : mem(at) {
    lane = threadIdx.x & 31, col = lane / Q, sub = lane % Q;
    seg_room = segments | 1;
    cores = reinterpret_cast<u32 *>(mem + rows * kRow);
    segs = cores + kTileCores * kSets;
    ord = reinterpret_cast<unsigned char *>(segs + ((KINDS & kKindRr) ? kSets * seg_room : 0));
    lst = ord + rows * kSets;
    goff = lst + ((KINDS & kKindGcaps) ? rows * kSets : 0);
  }
  __device__ __forceinline__ uint4 &own_at(int i, int c) const { return reinterpret_cast<uint4 *>(mem + i * kRow)[c]; }
  __device__ __forceinline__ float &inv_at(int i, int c) const { return reinterpret_cast<float *>(mem + i * kRow + kInv)[c]; }
  __device__ __forceinline__ int &priority_at(int i, int c) const { return reinterpret_cast<int *>(mem + i * kRow + kX)[c]; }
  __device__ __forceinline__ float &x(int i) const { return reinterpret_cast<float *>(mem + i * kRow + kX)[lane]; }
  __device__ __forceinline__ float &y(int i) const { return reinterpret_cast<float *>(mem + i * kRow + kY)[lane]; }

  // ---- for the stage: columns ------------------------------------------------------------------------
  __device__ __forceinline__ i64 most_gsegs() const {  // one more than a taskset may have
    const int room = (KINDS & kKindRr) ? seg_room + 1 : 64 * 32;
    return (KINDS & kKindRr) && room > 256 ? 256 : room;
  }
  __device__ __forceinline__ void keep_segment(int c, u32 k, u32 e) const {
    if (KINDS & kKindRr) segs[c * seg_room + (int)k] = e;
  }
  __device__ __forceinline__ void keep(const KParams &, int i, int c, u32 T, u32 D, u32 core, u32 segments, u32 first, u32 A,
                                       u32 Ge, u32, int priority) const {
    own_at(i, c) = make_uint4(tile_word(T, segments, core), __float_as_uint((float)D), __float_as_uint((float)A),
                              __float_as_uint((float)Ge) | (segments > 0 ? 0x80000000u : 0u));
    inv_at(i, c) = __frcp_rn((float)T);
    priority_at(i, c) = priority;
    if (KINDS & kKindRr) goff[i * kSets + c] = (unsigned char)first;
  }
  // ---- for the order: this lane's column ---------------------------------------------------------------
  __device__ __forceinline__ int priority(int i) const { return priority_at(i, col); }
  __device__ __forceinline__ u32 word(int i) const { return own_at(i, col).x; }
  __device__ __forceinline__ u32 &on_core(u32 core) const { return cores[(int)core * kSets + col]; }
  __device__ __forceinline__ unsigned char &order(int r) const { return ord[r * kSets + col]; }
  __device__ __forceinline__ void list_gpu(int n) const {
    int k = 0;
    for (int r = 0; r < n; ++r) {
      const int i = order(r);
      if (tile_segments(word(i)) != 0) lst[k * kSets + col] = (unsigned char)i, k += 1;
    }
  }
  // ---- for the walks -----------------------------------------------------------------------------------
  __device__ __forceinline__ float slices(int i, const uint4 &o, u32 L, u32 mode, u32 magic, u32 shift) const {
    const u32 *const e = segs + col * seg_room + goff[i * kSets + col];
    const int segments = (int)tile_segments(o.x);
    u32 sum = 0;
    for (int j = 0; j < segments; ++j) {
      const u32 w = e[j];
      sum += mode == 0 ? __umulhi(w + L - 1u, magic) >> shift : (mode == 1 ? w : (w > 0 ? 1u : 0u));
    }
    return (float)sum;
  }
};

// What a lane's walk is about.
struct KeptWalk {
  bool have;
  bool busy;    // the busy-waiting analysis
  float ovh;    // epsilon (GCAPS)
  float slot;   // L + theta (RR)
  u32 L, l_mode, l_magic, l_shift;
  i64 *out;     // results of the taskset, or null
};

// The taskset of this lane's column under this lane's analysis; as tile_walk, with the lemma set chosen by data.
template <bool GCAPS, class Rows>
__device__ __forceinline__ int kept_walk(const Rows &rows, const KeptWalk &w, bool literal, int n, int n_rt, int n_gpu) {
  const f32x2 two23 = pack2(kTwo23, kTwo23), minus23 = pack2(-kTwo23, -kTwo23), zero = pack2(0.0f, 0.0f);
  const int col = rows.col;
  const float eps2 = 2.0f * w.ovh;
  float g_sum = 0.0f;          // of all W^g
  u32 done = 0, gpu_done = 0;  // positions bounded so far, GPU-using ones among them
  bool alive = w.have && n > 0;
  int how = GCAPS_SCHED_YES, ended = n_rt;
  auto slots_of = [&](float slices) -> float { return slices == 0.0f ? 0.0f : fminf(w.slot * slices, (float)kFastClamp); };
#pragma unroll 1
  for (int r = 0;; ++r) {
    const bool active = alive && r < n_rt;
    const int n_list = __popc(gpu_done);
    // entries of the longest list, and one
    const int longest = GCAPS ? __reduce_max_sync(kFull, active ? n_list + 1 : 0) : (int)__any_sync(kFull, active);
    if (longest == 0) break;
    const int i = active ? rows.order(r) : 0;
    const uint4 own = rows.own_at(i, col);
    const u32 front = active ? rows.on_core(own.x >> 28) & done : 0u;
    const float T = tile_period(own.x), D = __uint_as_float(own.y), A = __uint_as_float(own.z);
    const float Ge = fabsf(__uint_as_float(own.w));
    const bool gi = (int)own.w < 0;
    float S, base;
    if (GCAPS) {
      const float eta = (float)tile_segments(own.x);
      S = eps2 * eta;
      base = A + Ge + S + (eta + 1.0f) * w.ovh;
    } else {
      float slices = 0.0f;
      if (active && gi) slices = rows.slices(i, own, w.L, w.l_mode, w.l_magic, w.l_shift);
      rows.y(i) = slices;
      S = slots_of(slices);
      base = A + Ge + (gi ? S * (float)(n_gpu - 1) : 0.0f);
    }
    const bool use_list = GCAPS && (w.busy || gi);
    const float nu = (float)(n_gpu - __popc(front & gpu_done) + 1);
    const int most_front = __reduce_max_sync(kFull, __popc(front));
    float R = base;
    bool go = active && !(R > D);
    auto gcaps_entry = [&](int h, bool have, f32x2 &I, f32x2 &J, f32x2 &W) {
      const uint4 o = rows.own_at(h, col);
      const float S_h = eps2 * (float)tile_segments(o.x), wg = w.busy ? fabsf(__uint_as_float(o.w)) + S_h : S_h;
      const float inv = have ? rows.inv_at(h, col) : 0.0f;
      I = pack2(inv, inv), J = pack2(rows.x(h), rows.y(h));
      W = pack2(have ? __uint_as_float(o.z) + wg : 0.0f, have && use_list ? -wg : 0.0f);
    };
    auto rr_entry = [&](int h, bool have, float &inv, float &j, float &weight) {
      const float A_h = __uint_as_float(rows.own_at(h, col).z);
      inv = have ? rows.inv_at(h, col) : 0.0f, j = rows.x(h);
      weight = have ? (w.busy ? fmaf(slots_of(rows.y(h)), nu, A_h) : A_h) : 0.0f;
    };
    auto list_pair = [&](int q, f32x2 &I, f32x2 &J, f32x2 &W) {
      float inv[2], j[2], weight[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const bool have = 2 * q + k < n_list;
        const int h = have ? rows.lst[(2 * q + k) * Rows::kSets + col] : 0;
        const uint4 o = rows.own_at(h, col);
        inv[k] = have ? rows.inv_at(h, col) : 0.0f, j[k] = rows.y(h);
        weight[k] = have ? fabsf(__uint_as_float(o.w)) + eps2 * (float)tile_segments(o.x) : 0.0f;
      }
      I = pack2(inv[0], inv[1]), J = pack2(j[0], j[1]), W = pack2(weight[0], weight[1]);
    };
    auto term = [&](f32x2 RR, f32x2 I, f32x2 J, f32x2 W, f32x2 acc) -> f32x2 {
      return fma2(add2(fma2_down(add2(RR, J), I, two23), minus23), W, acc);
    };
    auto run = [&](auto nc_tag, auto nl_tag, auto more_tag) {
      constexpr int NC = nc_tag, NL = GCAPS ? (int)nl_tag : 0, NX = GCAPS ? NC : NC / 2;
      constexpr bool MORE = more_tag;
      f32x2 CI[NX + 1], CJ[NX + 1], CW[NX + 1], LI[NL + 1], LJ[NL + 1], LW[NL + 1];
      u32 rest = front;
      f32x2 once = zero;
#pragma unroll
      for (int q = 0; q < NX; ++q) {
        const bool have = rest != 0;
        const int h = have ? __ffs((int)rest) - 1 : i;
        rest &= rest - 1u;
        if (GCAPS) {
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
      for (int q = 0; q < NL; ++q) list_pair(q, LI[q], LJ[q], LW[q]);
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
            if (GCAPS) {
              gcaps_entry(h, have, I, J, W);
            } else {
              float i0, j0, w0;
              rr_entry(h, have, i0, j0, w0);
              I = pack2(i0, 0.0f), J = pack2(j0, 0.0f), W = pack2(w0, 0.0f);
            }
            acc = term(RR, I, J, W, acc);
          }
          if (GCAPS) {
#pragma unroll 2
            for (int q = NL; 2 * q + 1 < longest; ++q) {
              f32x2 I, J, W;
              list_pair(q, I, J, W);
              list = term(RR, I, J, W, list);
            }
          }
        }
        float next = base + sum2(add2(acc, acc2));
        if (GCAPS) next += use_list ? sum2(add2(list, list2)) : 0.0f;
        const bool moved = go && next != R;
        R = moved ? next : R;
        go = moved && !(R > D);
      }
    };
    const int most_list = GCAPS ? longest >> 1 : 0;  // pairs
    if (!GCAPS && most_front == 0) {
      // (R = base)
      go = false;
    } else if (most_front <= 2 && most_list <= 2) {
      run(ModeTag<2>(), ModeTag<2>(), ModeTag<0>());
    } else if (most_front <= 4 && most_list <= 4) {
      run(ModeTag<4>(), ModeTag<4>(), ModeTag<0>());
    } else if (most_front <= 6 && most_list <= 6) {
      run(ModeTag<6>(), ModeTag<6>(), ModeTag<0>());
    } else if (GCAPS && most_front <= 6 && most_list <= 9) {
      run(ModeTag<6>(), ModeTag<9>(), ModeTag<0>());
    } else {
      run(ModeTag<6>(), ModeTag<6>(), ModeTag<1>());
    }
    if (active) {
      if (R > D || go) {  // a miss; a taskset that has used up its sweeps is left over (their limit is part of the result)
        if (w.out) w.out[i] = GCAPS_WCRT_MISS;
        alive = false, ended = r + 1;
        how = R > D ? GCAPS_SCHED_NO : -1;
      } else {
        if (w.out) w.out[i] = (i64)(int)R;
        const float t = T - 0.5f;
        if (GCAPS) {
          rows.x(i) = !w.busy && gi ? (R - A) + t : t, rows.y(i) = (R - Ge) + t;
          g_sum += gi ? Ge + S : 0.0f;
        } else {
          rows.x(i) = !w.busy && (gi || literal) ? (R - A) + t : t;
        }
        done |= 1u << i, gpu_done |= gi ? 1u << i : 0u;
      }
    }
  }
  if (GCAPS && w.out && w.have)
    for (int r = ended; r < n; ++r) w.out[rows.order(r)] = r < n_rt ? GCAPS_WCRT_SKIPPED : GCAPS_WCRT_BEST_EFFORT;
  return how;
}

// All walks of a tile.  False in the lane of a taskset that is left over.
template <int KINDS, int Q>
__device__ __forceinline__ bool kept_walks(const KParams &p, const SweepArgs &sw, const KeptRows<KINDS, Q> &rows, const TileLane &me) {
  typedef KeptRows<KINDS, Q> Rows;
  const int lane = rows.lane;
  const bool best_effort = (p.policy & GCAPS_RTA_BEST_EFFORT) != 0, literal = (p.policy & GCAPS_RTA_LITERAL) != 0;
  int n = __shfl_sync(kFull, me.n, rows.col);
  const i64 a = __shfl_sync(kFull, me.a, rows.col);
  const u32 t = __shfl_sync(kFull, me.t, rows.col);
  int n_rt = 0, n_gpu = 0;
  bool fits = true;
  if (rows.sub == 0) {
    fits = tile_order(rows, n, best_effort, n_rt, n_gpu);
    if (KINDS & kKindGcaps) rows.list_gpu(n);
  }
  fits = tile_worth(rows.sub == 0 && n > 0, fits);
  if (!fits) n = 0;
  n_rt = __shfl_sync(kFull, n_rt, rows.col * Q), n_gpu = __shfl_sync(kFull, n_gpu, rows.col * Q);
  __syncwarp();
  for (int i = 0; i < n; ++i) rows.x(i) = rows.y(i) = 0.0f;  // (finite, whatever else is there)
  bool all = fits;
  auto walks = [&](auto gcaps_tag) {
    constexpr bool GCAPS = gcaps_tag;
    const int first_mode = GCAPS ? 0 : 2;
    const int enabled = (sw.enabled >> first_mode) & 3;
    const int kinds = enabled == 3 ? 2 : 1, walks = enabled == 0 ? 0 : sw.n * kinds;
#pragma unroll 1
    for (int k0 = 0; k0 < walks; k0 += Q) {
      auto block_of = [&](int k, int &q, int &mode) {
        q = kinds == 2 ? k >> 1 : k, mode = first_mode + (enabled == 3 ? k & 1 : enabled >> 1);
        return q * sw.block_stride + sw.block_of_mode[mode];
      };
      int q, mode;
      const int k = k0 + rows.sub < walks ? k0 + rows.sub : k0;
      const int block = block_of(k, q, mode);
      const SweepPoint &pt = sw.q[q];
      KeptWalk w;
      w.have = k0 + rows.sub < walks, w.busy = (mode & 1) != 0, w.ovh = (float)(u32)pt.ovh;
      const u64 slot = (u64)pt.L + (u64)pt.ovh;
      w.slot = slot >= kFastClamp ? (float)kFastClamp : (float)(u32)slot;
      w.L = (u32)pt.L, w.l_mode = pt.l_mode, w.l_magic = pt.l_magic, w.l_shift = pt.l_shift;
      w.out = p.out_wcrt ? p.out_wcrt + (i64)block * p.n_tasks + a : nullptr;
      if (!GCAPS && p.out_wcrt) {
#pragma unroll 1
        for (int s = 0; s < Q && k0 + s < walks; ++s) {
          int q_s, mode_s;
          tile_fill(p.out_wcrt + (i64)block_of(k0 + s, q_s, mode_s) * p.n_tasks, me, lane);
        }
        if (w.have)
          for (int r = n_rt; r < n; ++r) w.out[rows.order(r)] = GCAPS_WCRT_BEST_EFFORT;
      }
      const int how = kept_walk<GCAPS>(rows, w, literal, n, n_rt, n_gpu);
      if (w.have && n > 0 && how >= 0) p.out_sched[(i64)block * p.n_tasksets + t] = (unsigned char)how;
      all &= !w.have || how >= 0;
    }
  };
  if (KINDS & kKindGcaps) walks(ModeTag<1>());
  if (KINDS & kKindRr) walks(ModeTag<0>());
  const u32 left = __ballot_sync(kFull, !all);
  __syncwarp();
  return lane >= Rows::kSets || ((left >> (lane * Q)) & ((1u << Q) - 1u)) == 0;
}

// sw.enabled: the analyses that run, all of KINDS.
template <int KINDS, int Q>
__global__ void __launch_bounds__(kTileThreads, Q == 2 ? 12 : 16)
rta_tile_kept_kernel(KParams p, int n, int segments, const __grid_constant__ SweepArgs sw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  let_dependents_start();  // (the launches behind this one wait for what it leaves over)
  const KeptRows<KINDS, Q> rows(smem_raw, tile_rows(n), segments);
  auto walk = [&](const TileLane &me) -> bool { return kept_walks<KINDS, Q>(p, sw, rows, me); };
  run_tiles<false>(p, n, rows, walk);
}

template <int KINDS, int Q>
cudaError_t launch_kept(const KParams &p, const SweepArgs &sw, int n, int sm_count, cudaStream_t st) {
  static int blocks_by_registers[64] = {0};
  // room for half as many GPU segments again as the batch has on average
  const double mean = (double)p.n_gsegs / (double)p.n_tasksets;
  const int segments = (KINDS & kKindRr) ? (mean > 160.0 ? 255 : (int)(1.5 * mean) + 8) : 0;
  const size_t smem = KeptRows<KINDS, Q>::bytes(tile_rows(n), segments);
  return launch_staged<kTileThreads>(false, rta_tile_kept_kernel<KINDS, Q>, blocks_by_registers,
                                     KeptRows<KINDS, Q>::bytes(32, 255), smem, kSmemPerSm / (smem + 1024), p.n_tasksets,
                                     sm_count, st, p, n, segments, sw);
}

}  // namespace
#endif  // GCAPS_RTA_TILE_KEPT_CUH_
