// gcaps_rta_tile.cu -- one analysis of small tasksets of one size, in tiles (rta_tile.cuh).
#include "rta_device.cuh"
#include "rta_tile.cuh"

using namespace gcaps_detail;

namespace {

// A tile of tasksets per warp.
template <int MODE>
__global__ void __launch_bounds__(kTileThreads, MODE < 2 ? 9 : 12) rta_tile_kernel(KParams p, int n) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  let_dependents_start();  // (the launches behind this one wait for what it leaves over)
  const TileRows<MODE> rows(smem_raw, tile_rows(n));
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
  run_tiles<(MODE >= 2)>(p, n, rows, walk);
}

template <int MODE>
cudaError_t launch_tile(const KParams &p, int n, int sm_count, cudaStream_t st) {
  static int blocks_by_registers[64] = {0};
  const size_t smem = TileRows<MODE>::bytes(tile_rows(n));
  return launch_staged<kTileThreads>(false, rta_tile_kernel<MODE>, blocks_by_registers, TileRows<MODE>::bytes(32), smem,
                                     kSmemPerSm / (smem + 1024), p.n_tasksets, sm_count, st, p, n);
}

}  // namespace

namespace gcaps_detail {

cudaError_t launch_tiles(int mode, const KParams &p, int n, int sm_count, cudaStream_t st) {
  switch (mode) {
    case 0: return launch_tile<0>(p, n, sm_count, st);
    case 1: return launch_tile<1>(p, n, sm_count, st);
    case 2: return launch_tile<2>(p, n, sm_count, st);
    case 3: return launch_tile<3>(p, n, sm_count, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace gcaps_detail
