// Storage of H and Ht as the tiles that the warp-specialised sensing kernel streams (sense_tc.cu), host-visible so that
// it can be enumerated without a GPU.
//
// A matrix of floats with rows of tile_kp(width) is cut into tiles of 128 rows (the last may have fewer) and a tile
// into chunks of SK floats of every row (the last chunk of a short row may be narrower), each contiguous, in the order
// in which a CTA streams them: a chunk is one bulk copy.  Rows of 8 chunks and more are padded with zeros to whole
// chunks, which spares the kernel the narrow ones (forward product of 48 transmitters, 130 receivers, 46^3: 95 against
// 97 us).  Short rows are not: receivers are the row length of Ht, and two of them padded to a chunk made it eight
// times as large.  Within a chunk the rows' parts follow each other; 16-byte piece j of row r lies at j ^ tile_swz, so
// that 8 threads that read the same piece of 8 rows from shared memory hit distinct banks (an odd number of pieces
// does so by itself; six meet in pairs).
#pragma once

namespace cisor {

#ifdef __CUDACC__
#define CISOR_TILE_HD __host__ __device__ __forceinline__
#else
#define CISOR_TILE_HD inline
#endif

constexpr int SK = 32;  // K (floats) per chunk

// floats from row to row (width is a multiple of 4)
CISOR_TILE_HD long long tile_kp(long long width) { return width < 8 * SK ? width : (width + SK - 1) / SK * SK; }
CISOR_TILE_HD int tile_swz(int r, int pieces) {
  return pieces == 8 ? r & 7 : pieces == 4 ? (r >> 1) & 3 : pieces == 2 ? (r >> 2) & 1 : 0;
}
// floats a row of the chunk that has `left` floats of the row to go
CISOR_TILE_HD int tile_width(long long left) { return left < SK ? (int)left : SK; }
// offset of chunk c of the tile from row r0 (a multiple of 128)
CISOR_TILE_HD int tile_rows(long long r0, long long rows) { return rows - r0 < 128 ? (int)(rows - r0) : 128; }
CISOR_TILE_HD long long tile_chunk(long long r0, long long c, long long rows, long long kp) {
  return r0 * kp + c * (tile_rows(r0, rows) * SK);
}
// within a chunk: offset of 16-byte piece j of row r
CISOR_TILE_HD int tile_piece(int r, int j, int pieces) { return (r * pieces + (j ^ tile_swz(r, pieces))) * 4; }
// offset of element k of a row, kp = tile_kp(width)
CISOR_TILE_HD long long tile_off(long long row, long long k, long long rows, long long kp) {
  const long long r0 = row & ~127ll, c = k / SK;
  return tile_chunk(r0, c, rows, kp) + tile_piece((int)(row - r0), (int)(k & (SK - 1)) >> 2, tile_width(kp - c * SK) >> 2) +
         (k & 3);
}

}  // namespace cisor
