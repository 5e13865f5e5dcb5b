// Host check of row_tiles.h, run by tests/test_row_tiles.py.
#include <cstdio>
#include <vector>

#include "../../paper_1104_1703_gb300/csrc/row_tiles.h"

using gbmg::RowTiles;

static int fails = 0;

static void check(int nx, int ny, int nz, int cells, int warps) {
  const RowTiles T = gbmg::row_tiles(nx, ny, nz, cells, warps);
  // every cell in exactly one tile, in order, at the row and place it says
  unsigned long long at = 0;
  for (unsigned t = 0; t < T.count; ++t) {
    unsigned row, i0, n;
    T.tile(t, &row, &i0, &n);
    if (n < 1 || n > (unsigned)cells || (unsigned long long)row * nx + i0 != at) ++fails;
    for (unsigned c = 0; c < n; ++c) {
      const unsigned dr = T.per > 1 ? T.row_of(c) : 0u;
      if (((unsigned long long)(row + dr) * nx + (i0 + c - dr * nx)) != at + c || i0 + c - dr * nx >= (unsigned)nx) ++fails;
    }
    at += n;
  }
  if (at != (unsigned long long)nx * ny * nz) ++fails;
  // no more warp rounds of 32 cells than a flat walk over the cells (or one per
  // warp) takes, up to the ends of tiles (below twice as many)
  unsigned long long rounds = 0;
  for (unsigned t = 0; t < T.count; ++t) {
    unsigned row, i0, n;
    T.tile(t, &row, &i0, &n);
    rounds += (n + 31) / 32;
  }
  const unsigned long long flat = (at + 31) / 32;
  const unsigned long long enough = flat > (unsigned long long)warps ? flat : warps;
  if (rounds > 2 * enough + 1) {
    ++fails;
    std::printf("%d x %d x %d, tiles of %d: %llu rounds, flat %llu\n", nx, ny, nz, cells, rounds, flat);
  }
}

int main() {
  for (int cells : {128, 256})
    for (int nx = 1; nx <= 2048; ++nx) {
      check(nx, 3, 5, cells, 64);
      check(nx, 37, 11, cells, 8);
      if (nx <= 300) check(nx, 64, 50, cells, 16);
      if (nx <= 8) check(nx, 1024, 1024, cells, 9728);
    }
  check(2048, 2048, 1, 256, 9728);
  check(1, 2048, 2048, 256, 9728);
  std::printf(fails ? "%d failures\n" : "ok\n", fails);
  return fails != 0;
}
