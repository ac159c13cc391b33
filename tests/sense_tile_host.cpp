// Host enumeration of csrc/sense_tile.cuh.  For every shape: the elements fill [0, rows kp) exactly once, kp within
// an eighth of the width; a chunk of
// a tile is contiguous, starts on 16 bytes at tile_chunk and holds the pieces where the kernel looks for them
// (tile_piece); 8 rows' equal pieces, as 8 threads read them, lie in distinct banks (six pieces a row: at most two
// together).  Prints the number of violations.
#include <cstdio>
#include <vector>

#include "sense_tile.cuh"

using namespace cisor;

int main() {
  long bad = 0;
  const long long rows_of[] = {1, 2, 7, 36, 127, 128, 129, 300}, width_of[] = {4, 8, 12, 16, 20, 24, 28, 32, 36, 72, 92, 128, 252, 256, 260, 720};
  for (long long rows : rows_of)
    for (long long width : width_of) {
      const long long kp = tile_kp(width);
      if (kp < width || kp > width + width / 8) ++bad;
      std::vector<char> seen(rows * kp, 0);
      for (long long r = 0; r < rows; ++r)
        for (long long k = 0; k < kp; ++k) {
          const long long o = tile_off(r, k, rows, kp);
          if (o < 0 || o >= rows * kp || seen[o]++) {
            ++bad;
            continue;
          }
          const long long r0 = r / 128 * 128, c = k / SK, base = tile_chunk(r0, c, rows, kp);
          const int R = tile_rows(r0, rows), w = tile_width(kp - c * SK);
          if (base % 4 || w % 4 || o < base || o >= base + (long long)R * w) ++bad;
          if (o != base + tile_piece((int)(r - r0), (int)(k % SK) / 4, w / 4) + k % 4) ++bad;
        }
    }
  for (int pieces = 1; pieces <= 8; ++pieces)
    for (int r0 = 0; r0 < 128; r0 += 8)
      for (int j = 0; j < pieces; ++j) {
        int hit[8] = {};
        for (int r = r0; r < r0 + 8; ++r)
          if (++hit[tile_piece(r, j, pieces) / 4 % 8] > (pieces == 6 ? 2 : 1)) ++bad;
      }
  std::printf("%ld\n", bad);
  return 0;
}
