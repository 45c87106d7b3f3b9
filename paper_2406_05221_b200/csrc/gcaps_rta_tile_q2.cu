// gcaps_rta_tile_q2.cu -- tiles whose tasksets have 2 lanes each, one per analysis and (timeslice, overhead) pair.
#include "rta_device.cuh"
#include "rta_tile_kept.cuh"

namespace gcaps_detail {

cudaError_t launch_tile_q2(const KParams &p, const SweepArgs &sw, int n, int sm_count, cudaStream_t st) {
  if ((sw.enabled & 12) == 0) return launch_kept<kKindGcaps, 2>(p, sw, n, sm_count, st);
  if ((sw.enabled & 3) == 0) return launch_kept<kKindRr, 2>(p, sw, n, sm_count, st);
  return launch_kept<kKindGcaps | kKindRr, 2>(p, sw, n, sm_count, st);
}

}  // namespace gcaps_detail
