// Which tiles a warp looks at (csrc/tile_patience.h): a row of tiles, '.' for one that a walk takes and 'x' for one whose tasksets
// are all left over; prints for each tile 'l' if it is looked at, '-' if not.
//   tile_patience_host ROW
#include "../paper_2406_05221_b200/csrc/tile_patience.h"

#include <cstdio>

int main(int argc, char **argv) {
  if (argc != 2) return 2;
  TilePatience patience = {0};
  for (const char *tile = argv[1]; *tile; ++tile) {
    const bool looks = patience.looks();
    patience.done(!looks || *tile == 'x' ? 32 : 7, 32);
    std::putchar(looks ? 'l' : '-');
  }
  return 0;
}
