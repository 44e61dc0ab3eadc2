// Where the query tiles of k_attn_tc come from: the shape of the tensor map over the query rows and the coordinates of a tile in it.
// Plain C++ but for one function's qualifier, so that the fetched addresses can be checked without a GPU.
#pragma once

#ifdef __CUDACC__
#define Q_TILE_FN __host__ __device__ static __forceinline__
#else
#define Q_TILE_FN static inline
#endif

// Five dimensions, innermost first: elements (strides in bytes, the innermost is 2) and the box of a copy.
struct QTileMap { unsigned long long dims[5], strides[4]; unsigned box[5]; };

// The query rows [rows][H][high | low][hd] as the tiles take them: eight entries' high parts, then their low parts, then the next
// eight entries.  With G heads per KV head an eight is rpg = 8 / G rows of G heads, or eight heads of one row; the box is the whole
// 128-row tile either way.  In the first form a row enters through two dimensions, row within an eight (2) and eight (4), and
// a tile that starts c2 rows into an eight takes rows c2 .. c2 + rpg - 1 of each.  Eights behind the last are cut off, so what a
// tile reads behind `rows` is the last eight's c2 <= rpg - 1 rows: q_tile_room.  (Both dimensions as plain rows, which needs no c2, cuts nothing off:
// up to 56 rows behind the buffer were read, where other CTAs of the launch store their outputs.)
static inline QTileMap q_tile_map(int rows, int H, int G, int hd) {
  const unsigned long long part = (unsigned long long)hd * 2, head = part * 2, row = head * H, r = (unsigned long long)rows, h = (unsigned long long)H;
  if (G <= 8) {
    const unsigned rpg = 8u / (unsigned)G;
    return QTileMap{{(unsigned long long)hd, h, 2ull * rpg - 1ull, 2ull, (r + rpg - 1) / rpg}, {head, row, part, row * rpg}, {64u, (unsigned)G, rpg, 2u, 8u}};
  }
  return QTileMap{{(unsigned long long)hd, h, 2ull, (unsigned long long)(G / 8), r}, {head, part, head * 8, row}, {64u, 8u, 2u, (unsigned)(G / 8), (unsigned)(64 / G)}};
}

// Coordinates 2 and 4 of the tile that starts at query row `row` (0 and 1 are the column and the first head, 3 is 0).
Q_TILE_FN void q_tile_start(int G, int row, int &c2, int &c4) {
  const int lg = G >= 8 ? 0 : G == 4 ? 1 : G == 2 ? 2 : 3;      // log2(8 / G)
  c2 = row & ((1 << lg) - 1);
  c4 = row >> lg;
}

// Rows that a buffer of `rows` query rows (a multiple of 8) has room for: behind them the rows that tiles read and nobody uses.
// A prompt's tiles start on whole eights and read none.
static inline int q_tile_room(int rows) { return rows + 7; }
