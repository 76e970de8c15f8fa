"""The deposit's bin arrays hold the bins of every tile shape that a context takes, on every mesh
side: the host geometry (csrc/bin_geo.h) compiled here and checked shape by shape, no GPU."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2211_09815_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "bin_geo.h"
int main() {
  int shapes = 0;
  for (int lg = 3; lg <= 10; ++lg) {
    long long most = 0;
    for (int z = 0; z <= 12; ++z)
      for (int y = 0; y <= 12; ++y)
        for (int x = 0; x <= 12; ++x) {
          const int l[3] = {z, y, x};
          if (!pmgb::tile_ok(l, 12)) continue;
          const pmgb::BinGeo bg = pmgb::make_bin_geo(lg, x, y, z);
          // tiles cover the mesh, eight bins each
          if ((long long)bg.ntiles << (bg.lx + bg.ly + bg.lz) != 1LL << (3 * lg) || bg.nkeys != 8LL * bg.ntiles) return 1;
          if (bg.nkeys > most) most = bg.nkeys;
          ++shapes;
        }
    std::printf("%d %lld %lld\n", 1 << lg, most, pmgb::max_bin_keys(lg));
  }
  // the default shapes: 2^10 cells where a mesh makes few tiles, else 2^12 and 2^11
  const int def[4][3] = {{2, 2, 6}, {3, 4, 5}, {2, 2, 6}, {2, 3, 6}};
  for (int k = 0; k < 4; ++k)
    if (!pmgb::tile_ok(def[k], k < 2 ? 12 : 11)) return 2;
  return shapes ? 0 : 3;
}
"""


def test_every_tile_shape_fits_the_bin_arrays(tmp_path):
    src, exe = tmp_path / "bins.cpp", tmp_path / "bins"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    rows = [tuple(int(v) for v in line.split()) for line in out.splitlines()]
    assert [r[0] for r in rows] == [8, 16, 32, 64, 128, 256, 512, 1024]
    for side, most, allocated in rows:
        assert most == allocated, side   # enough, and no more than the worst shape needs
