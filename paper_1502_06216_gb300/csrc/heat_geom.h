// heat_geom.h -- geometry of the heat kernel's resident tiles (heat_tile.cu): which block
// owns which cells, which cells it sends and for which it waits.  Plain C++ for both sides,
// so that the relation "waits for" can be enumerated without a GPU.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>

#ifndef JKO_HD
#ifdef __CUDACC__
#define JKO_HD __host__ __device__ __forceinline__
#else
#define JKO_HD inline
#endif
#endif

namespace jko {
namespace heat_geom {

constexpr int H = 4;   // cells of the halo, and Clenshaw steps per exchange at most

// flags of a cell of a tile's box: free, and its four neighbours'; inside the grid
enum : int { FREE = 1, LEFT = 2, RIGHT = 4, UP = 8, DOWN = 16, IN_GRID = 32 };

JKO_HD bool in_grid(int x, int y, int nx, int ny) { return x >= 0 && x < nx && y >= 0 && y < ny; }
JKO_HD bool is_free(int x, int y, int nx, int ny, const uint8_t* mask) {
  return in_grid(x, y, nx, ny) && (mask == nullptr || mask[(size_t)y * nx + x] == 0);
}
JKO_HD int cell_flags(int x, int y, int nx, int ny, const uint8_t* mask) {
  if (!in_grid(x, y, nx, ny)) return 0;
  if (!is_free(x, y, nx, ny, mask)) return IN_GRID;
  return IN_GRID | FREE | (is_free(x - 1, y, nx, ny, mask) ? LEFT : 0) |
         (is_free(x + 1, y, nx, ny, mask) ? RIGHT : 0) | (is_free(x, y - 1, nx, ny, mask) ? UP : 0) |
         (is_free(x, y + 1, nx, ny, mask) ? DOWN : 0);
}

// The cells of one block.
struct Tile {
  int x0, y0, w, h;
};
JKO_HD Tile tile_of(int block, int tw, int th, int ntx, int nx, int ny) {
  const int by = block / ntx, bx = block - by * ntx;
  Tile t{bx * tw, by * th, tw, th};
  if (t.x0 + tw > nx) t.w = nx - t.x0;
  if (t.y0 + th > ny) t.h = ny - t.y0;
  return t;
}

// The ring of H cells around a tile: its cells, and the place of cell i in the tile's box
// (the tile at (H, H)); inv_bx = 1 / (w + 2 H).
JKO_HD int ring_cells(const Tile& t) { return 2 * H * (t.w + 2 * H) + 2 * H * t.h; }
JKO_HD void ring_place(int i, const Tile& t, float inv_bx, int& ex, int& ey) {
  const int BX = t.w + 2 * H, top = 2 * H * BX;
  if (i < top) {
    const int r = (int)(((float)i + 0.5f) * inv_bx);   // i / BX (exact below 2^20)
    ex = i - r * BX;
    ey = r < H ? r : t.h + r;
  } else {
    i -= top;
    const int r = i / (2 * H), col = i - r * 2 * H;
    ex = col < H ? col : t.w + col;
    ey = H + r;
  }
}

// The cells a block sends (cell (x, y) of its tile) and those of its ring it waits for: all
// of the grid, masked ones too (their iterates are zeros).  Then block a waits for block b
// exactly where a cell of b lies within H cells of a's tile, which is symmetric; waiting for
// free cells alone is not (a tile whose edge is all obstacle would be read and never waited
// for, and its neighbour could overwrite words it has yet to read).
JKO_HD bool sent(int x, int y, const Tile& t) {
  return x < H || x >= t.w - H || y < H || y >= t.h - H;
}
JKO_HD bool awaited(int flags) { return flags & IN_GRID; }

// Shared memory of a block: three FP64 images and the flags over the tile's box, four images of
// `es` bytes an element over the tile.
JKO_HD size_t tile_bytes(int tw, int th, size_t es) {
  const size_t box = (size_t)(tw + 2 * H) * (th + 2 * H);
  return box * 25 + (size_t)tw * th * es * 4;
}

// The tile shape for at most `blocks` blocks: the least work of a phase of H steps, in warps.
inline void tile_shape(int nx, int ny, int blocks, int* tw, int* th) {
  long long best = -1;
  for (int gx = 1; gx <= std::min(nx, blocks); ++gx) {
    const int gy = std::min(ny, blocks / gx);
    const int w = (nx + gx - 1) / gx, h = (ny + gy - 1) / gy;
    long long c = 0;
    for (int e = 0; e < H; ++e) c += ((long long)(w + 2 * e) * (h + 2 * e) + 31) / 32;
    if (best < 0 || c < best) {
      best = c;
      *tw = w;
      *th = h;
    }
  }
}

}  // namespace heat_geom
}  // namespace jko
