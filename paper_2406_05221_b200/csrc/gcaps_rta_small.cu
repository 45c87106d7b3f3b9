// gcaps_rta_small.cu -- one analysis of tasksets of up to 32 tasks, with a plan: tiles of tasksets, and the
// kernel that takes what no tile takes.
#include "rta_device.cuh"
#include "rta_tile.cuh"

using namespace gcaps_detail;

namespace {

// The bins of up to 32 tasks in one persistent launch, largest tasksets first: (lanes per
// taskset, tasks per lane) = (16,2) (8,3) (8,2) (8,1) for at most 32, 24, 16, 8 tasks, i.e. two or
// four tasksets per warp.  (A look at the first ranks out of a stage, a warp per taskset, was slower
// here in every form tried: 100,000 24-task tasksets under round robin 163 us against 128.)
template <int MODE>
__global__ void __launch_bounds__(kBlockThreads, min_blocks(3)) rta_small_kernel(KParams p, bool rest) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (rest) wait_for_previous_grid();  // what the tiles left over is listed from here on
  let_dependents_start();  // the kernel of the next size bin shares no data with this one
  u32 *warp_buf = reinterpret_cast<u32 *>(smem_raw) + (threadIdx.x >> 5) * kSmallWarpWords;
  Ahead *ahead = reinterpret_cast<Ahead *>(warp_buf + kSmallWarpWords - kAheadWords);
  run_bin<16, 2, 1 << MODE>(p, 3, warp_buf, ahead);
  run_bin<8, 3, 1 << MODE>(p, 2, warp_buf, ahead);
  run_bin<8, 2, 1 << MODE>(p, 1, warp_buf, ahead);
  run_bin<8, 1, 1 << MODE>(p, 0, warp_buf, ahead);
  wait_for_previous_grid();
}

// A tile of tasksets per warp; n_rows: positions that tiles have room for.
template <int MODE>
__global__ void __launch_bounds__(kTileThreads, MODE < 2 ? 9 : 12) rta_tile_kernel(KParams p, int n_rows) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  let_dependents_start();  // (the launches behind this one wait for what it leaves over)
  const TileRows<MODE> rows(smem_raw, n_rows);
  const float ovh = (float)(u32)p.ovh;
  const bool literal = (p.policy & GCAPS_RTA_LITERAL) != 0;
  auto walk = [&](const TileLane &me) -> bool {
    int n_rt, n_gpu;
    const bool few = tile_order(rows, me.n, (p.policy & GCAPS_RTA_BEST_EFFORT) != 0, n_rt, n_gpu);
    const bool fits = tile_worth(me.n > 0, few);
    const int n = fits ? me.n : 0;
    rows.clear();
    if (MODE >= 2) {
      tile_fill(p.out_wcrt, me, threadIdx.x & 31);
      for (int r = n_rt; r < n; ++r) p.out_wcrt[me.a + rows.order(r)] = GCAPS_WCRT_BEST_EFFORT;
    }
    const int how = tile_walk<MODE>(rows, ovh, literal, n, n_rt, n_gpu, p.out_wcrt + me.a);
    if (n > 0 && how >= 0) p.out_sched[me.t] = (unsigned char)how;
    return fits && how >= 0;
  };
  run_tiles<(MODE >= 2)>(p, n_rows, rows, walk);
}

template <int MODE>
cudaError_t launch_tile(const KParams &p, int rows, int sm_count, cudaStream_t st) {
  static int blocks_by_registers[64] = {0};
  const size_t smem = TileRows<MODE>::bytes(rows);
  return launch_staged<kTileThreads>(false, rta_tile_kernel<MODE>, blocks_by_registers, TileRows<MODE>::bytes(32), smem,
                                     kSmemPerSm / (smem + 1024), p.n_tasksets, sm_count, st, p, rows);
}

template <int MODE>
cudaError_t launch_groups(const KParams &p, bool rest, int sm_count, cudaStream_t st) {
  constexpr int kWarps = kBlockThreads / 32;
  static int blocks_per_sm[64] = {0};
  return launch_persistent_ex(rest, rta_small_kernel<MODE>, blocks_per_sm, sizeof(u32) * kSmallWarpWords * kWarps,
                              (p.n_tasksets + kWarps - 1) / kWarps, sm_count, st, p, rest);
}

template <int MODE>
cudaError_t launch_small_mode(const KParams &p, int rows, int sm_count, cudaStream_t st) {
  if (rows == 0) return launch_groups<MODE>(p, false, sm_count, st);
  const cudaError_t e = launch_tile<MODE>(p, rows, sm_count, st);
  return e == cudaSuccess ? launch_groups<MODE>(p, true, sm_count, st) : e;
}

}  // namespace

namespace gcaps_detail {

// Tiles are for batches of tasksets of one size (a mean that is a whole number): a tile's rows are taken by the largest
// taskset, and in a mixture the plan's bins are the better way (4 to 24 tasks, 100,000 tasksets 212 us in tiles, 162
// us in bins).  Under GCAPS a tile's walk is long, so there have to be enough tiles to go round: 12 tasks 43 / 54 us (tiles /
// bins) at 12,500 tasksets and 63 / 84 at 50,000, 16 tasks 71 / 69 at 25,000 and 79 / 83 at 35,000, 20 tasks 91 / 84
// and 97 / 105, 24 tasks 127 / 123 at 35,000 and 128 / 157 at 50,000.  Under RR tiles are the faster way from the start
// (24 tasks 40 / 51 us at 12,500).  Several analyses under GCAPS, 20 tasks: 170 / 138 us for five pairs of 10,000
// tasksets, 243 / 240 of 20,000, 212 / 280 for three pairs of 50,000; 24 tasks: 203 / 182 for two pairs of 30,000, 578 / 654 for
// 25 pairs of 5,000.  32 tasks: 575 / 521 us per 100,000, as a tile then takes 40 KB.
int tile_rows(int analyses, int walks, i64 max_ovh, const KParams &p) {
  if (max_ovh >= (1 << 20) || ((analyses & 2) && (p.policy & GCAPS_RTA_LITERAL))) return 0;
  if (p.n_tasks % p.n_tasksets != 0 || p.n_tasks > 24 * p.n_tasksets) return 0;
  const int n = (int)(p.n_tasks / p.n_tasksets);
  if (walks == 1 && (analyses & 3) && n > 12 && p.n_tasksets < 1750 * n) return 0;
  if (walks > 1 && (analyses & 12) == 0 && n > 12 && p.n_tasksets * walks < 100000) return 0;
  return n < 4 ? 4 : n;
}

cudaError_t launch_small(int mode, const KParams &p, int rows, int sm_count, cudaStream_t st) {
  switch (mode) {
    case 0: return launch_small_mode<0>(p, rows, sm_count, st);
    case 1: return launch_small_mode<1>(p, rows, sm_count, st);
    case 2: return launch_small_mode<2>(p, rows, sm_count, st);
    case 3: return launch_small_mode<3>(p, rows, sm_count, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace gcaps_detail
