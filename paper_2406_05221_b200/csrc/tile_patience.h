/* tile_patience.h -- which of its tiles a warp looks at.  Plain C++ without CUDA: the kernels (rta_tile.cuh) use it, and a
 * host program can too. */
#ifndef GCAPS_TILE_PATIENCE_H_
#define GCAPS_TILE_PATIENCE_H_

#ifdef __CUDACC__
#define PATIENCE_FN __device__ __forceinline__
#else
#define PATIENCE_FN inline
#endif

constexpr int kTilesUnseen = 7;

/* Tasksets of a batch tend to be alike: a warp that walked a tile and had to leave three quarters of it to the launches behind all
 * the same leaves the next kTilesUnseen tiles too, without a look, and then looks again.  Tasksets that are left before the walk do not
 * count, as they cost little: warps that pass tiles by pull the next ones all the faster, and a stretch of such tasksets would take a
 * multiple of its length. */
struct TilePatience {
  int unseen; /* tiles still to be left without a look */
  PATIENCE_FN bool looks() const { return unseen == 0; }
  /* the tile in hand is done; `left` of its tasksets are left over after the walk */
  PATIENCE_FN void done(int left, int tasksets) {
    if (unseen > 0) unseen -= 1;
    else if (4 * left >= 3 * tasksets) unseen = kTilesUnseen;
  }
};

#endif /* GCAPS_TILE_PATIENCE_H_ */
