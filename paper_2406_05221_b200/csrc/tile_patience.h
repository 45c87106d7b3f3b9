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

/* Tasksets of a batch tend to be alike: a warp that had to leave three quarters of a tile to the launches behind leaves the
 * next kTilesUnseen tiles too, without a look, and then looks again. */
struct TilePatience {
  int unseen; /* tiles still to be left without a look */
  PATIENCE_FN bool looks() const { return unseen == 0; }
  /* the tile in hand is done; `left` of its tasksets are left over */
  PATIENCE_FN void done(int left, int tasksets) {
    if (unseen > 0) unseen -= 1;
    else if (4 * left >= 3 * tasksets) unseen = kTilesUnseen;
  }
};

#endif /* GCAPS_TILE_PATIENCE_H_ */
