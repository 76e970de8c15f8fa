// Tile geometry of the deposit bins (host code, also compiled by the CPU tests).
#pragma once

namespace pmgb {

// Bins of the tile-owner deposit (bin_kernels.cuh): mesh tiles of 2^lx x 2^ly x 2^lz cells
// (x = array axis 2), and per tile a class of three bits, set when the particle's cell is on
// the tile's last layer along x, y or z (its CIC cloud reaches into the next tile there).
struct BinGeo {
  int lx, ly, lz;       // log2 of the tile extent along axes 2, 1, 0
  int ntx, nty, ntz;    // tiles per axis
  int ntiles;           // per instance
  long long nkeys;      // bins per instance = 8 ntiles
};

// (extents longer than the mesh are cut to it)
inline BinGeo make_bin_geo(int lg_nm, int lx, int ly, int lz) {
  BinGeo b;
  b.lx = lx < lg_nm ? lx : lg_nm;
  b.ly = ly < lg_nm ? ly : lg_nm;
  b.lz = lz < lg_nm ? lz : lg_nm;
  b.ntx = 1 << (lg_nm - b.lx);
  b.nty = 1 << (lg_nm - b.ly);
  b.ntz = 1 << (lg_nm - b.lz);
  b.ntiles = b.ntx * b.nty * b.ntz;
  b.nkeys = 8LL * b.ntiles;
  return b;
}

// Tile shapes (log2 of z, y, x) a deposit takes: x at least 4 cells (vector write-out),
// 2^9..2^maxl cells (shared memory: 2^12 cells x 8 B for the density alone, 2^11 x 32 B with
// the pi sums)
inline bool tile_ok(const int* l, int maxl) {
  return l[0] >= 0 && l[1] >= 0 && l[2] >= 2 && l[0] + l[1] + l[2] >= 9 && l[0] + l[1] + l[2] <= maxl &&
         l[0] <= 10 && l[1] <= 10 && l[2] <= 10;
}

// Most bins per instance of any shape that tile_ok takes: what the bin arrays are sized for.
// A shape of 2^9 cells cut to a mesh of side 2^lg_nm keeps 2^min(9, lg_nm) of them at least
// (x = 2^9: one row), so that small meshes can have more, smaller tiles than 2^9 cells make.
inline long long max_bin_keys(int lg_nm) { return 8LL << (3 * lg_nm - (lg_nm < 9 ? lg_nm : 9)); }

}  // namespace pmgb
