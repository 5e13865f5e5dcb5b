// How the warps of a kernel that runs along the rows of an nx * ny * nz array
// (x fastest) share its cells: tiles of up to `cells` consecutive ones, parts
// of a row or, where rows are short, several whole rows, so that a tile's
// lanes have work for any nx.
#pragma once

#include <cuda_runtime.h>

namespace gbmg {

struct RowTiles {
  unsigned nx, rows;  // cells per row, rows (ny * nz) of the array
  unsigned cells;     // of a tile, at most
  unsigned parts;     // tiles per row; 1 if a tile has several rows
  unsigned per;       // rows per tile
  unsigned inv;       // c / nx = c * inv >> 16 for a tile's cell c
  unsigned count;

  // First row and first cell there of tile t, and the tile's cells.
  __host__ __device__ void tile(unsigned t, unsigned* row, unsigned* i0, unsigned* n) const {
    if (per > 1) {
      *row = t * per;
      *i0 = 0;
      const unsigned left = rows - *row;
      *n = (left < per ? left : per) * nx;
    } else {
      *row = t / parts;
      *i0 = (t - *row * parts) * cells;
      const unsigned left = nx - *i0;
      *n = left < cells ? left : cells;
    }
  }
  // Row (from the tile's first) of its cell c.
  __host__ __device__ unsigned row_of(unsigned c) const { return c * inv >> 16; }
};

// Rows of which two or more fit a tile (cells <= 256) are put together as far
// as that leaves each of `warps` warps a tile.
// (c * inv >> 16 with inv = 65536 / nx + 1 is the quotient: c * inv / 65536
// exceeds c / nx by at most c / 65536, less than the 1 / nx that it must stay
// under, as c nx <= cells * cells / 2 < 65536.)
inline RowTiles row_tiles(int nx, int ny, int nz, int cells, int warps) {
  RowTiles r;
  r.nx = (unsigned)nx;
  r.rows = (unsigned)ny * (unsigned)nz;
  r.cells = (unsigned)cells;
  r.inv = 65536u / r.nx + 1u;
  const unsigned fit = r.cells / r.nx, want = (r.rows + (unsigned)warps - 1) / (unsigned)warps;
  r.per = fit < want ? fit : want;
  if (r.per > 1) {
    r.parts = 1;
    r.count = (r.rows + r.per - 1) / r.per;
  } else {
    r.per = 1;
    r.parts = (r.nx + r.cells - 1) / r.cells;
    r.count = r.parts * r.rows;
  }
  return r;
}

}  // namespace gbmg
