"""How a Phase-3 launch's tiles are split over its CTAs, checked on the host (no GPU).

`TileRun` and `TileWalk` in `csrc/fw_kernels.cu` give every CTA its whole tiles
and, where left-over tiles are cut, its parts of the k-steps.  This test copies
their definitions out of the source unchanged, compiles them with g++ and walks
every CTA of many launches: each k-step of each tile has to be taken exactly
once, whatever the grid, the mode and the next-diagonal task.
"""
import os
import re
import shutil
import subprocess

import pytest

from tests.test_plan_source import CSRC, _block

MAIN = r"""
#include <cstdlib>
#include <cstdio>
#include <map>
template <class W> int walk(int tx, int ty, int sym, int epw, int chain, int grid, int &lp_max) {
  std::map<std::pair<int, int>, int> seen;  // (tile row, tile column) -> k-steps taken
  int tiles = 0;
  for (int y = 0; y < ty; ++y) tiles += tx - (sym ? std::min(tx, y / epw) : 0);
  gridDim.x = grid;
  for (blockIdx.x = 0; (int)blockIdx.x < grid; ++blockIdx.x) {
    W w;
    w.tiles_x = tx; w.tiles_y = ty; w.sym = sym;
    w.plan(tiles, chain);
    if (w.nu <= 0) continue;
    w.begin();
    for (int k = 0; k < w.nu; ++k) {
      if (w.ty < 0 || w.ty >= ty || w.tx >= tx || w.tx < (sym ? w.ty / epw : 0)) return 1;
      const int ks = w.ksteps(64);
      if (w.part * ks + ks > 64) return 2;
      seen[{w.ty, w.tx}] += (ks == 64) ? 64 : (1 << (w.part * 4)) * 1000;  // parts apart from whole tiles
      if (ks < 64) lp_max = std::max(lp_max, ks == 32 ? 1 : 2);
      w.next();
    }
  }
  if ((int)seen.size() != tiles) return 3;
  for (auto &s : seen)
    if (s.second != 64 && s.second != 17 * 1000 && s.second != (1 + 16 + 256 + 4096) * 1000) return 4;
  return 0;
}
int main() {
  int cut = 0, bad = 0;
  for (int grid : {1, 2, 3, 7, 38, 151, 152})
    for (int t = 1; t <= 44; ++t)
      for (int sym = 0; sym < 2; ++sym)
        for (int chain = 0; chain < 2; ++chain) {
          const int tiles = sym ? t * (t + 1) / 2 : t * t;
          int unused = 0;
          const int g1 = std::min(grid, tiles + chain), g2 = std::min(grid, 4 * tiles + chain);
          if (g2 - (((tiles + chain) / g2 == 0) ? chain : 0) <= 0) continue;
          int r = walk<TileRun<One>>(t, t, sym, 1, chain, g1, unused);
          if (!r) r = walk<TileRun<Two>>(t, 2 * t, sym, 2, chain, g1, unused);
          if (!r) r = walk<TileRun<One>>(t, t, sym, 1, chain, grid, unused);  // a grid sized for another mode
          if (!r) r = walk<TileWalk<One>>(t, t, sym, 1, chain, g2, cut);
          if (!r && grid > chain) r = walk<TileWalk<One>>(t, t, sym, 1, chain, grid, cut);
          if (r && !bad) { printf("grid %d tiles %d sym %d chain %d: %d\n", grid, t, sym, chain, r); bad = 1; }
          const double gain = split_gain(tiles, chain, grid);
          if (!(gain >= 0.0 && gain < 1.0)) { printf("gain %g\n", gain); bad = 1; }
        }
  printf("cut %d bad %d\n", cut, bad);
  return bad;
}
"""


def test_every_k_step_of_every_tile_is_taken_once(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ needed")
    ker = open(os.path.join(CSRC, "fw_kernels.cu")).read()
    prog = "\n".join([
        "#include <algorithm>", "#include <cstdint>", "using std::min; using std::max;",
        "#define __device__", "#define __host__", "#define __forceinline__ inline",
        "struct { unsigned x; } gridDim, blockIdx;",
        "struct One { static constexpr int EPW = 1; }; struct Two { static constexpr int EPW = 2; };",
        _block(ker, "long long sym_prefix(", with_template=False).replace("__device__", "static"),
        _block(ker, "struct TileGrid {"), _block(ker, "struct TileRun : "),
        re.search(r"constexpr int kPartCost = \d+;", ker).group(0),
        _block(ker, "int wave_parts(", with_template=False).replace("int wave_parts(", "inline int wave_parts(", 1),
        _block(ker, "struct TileWalk : "),
        _block(ker, "static double split_gain(", with_template=False), MAIN])
    src, exe = tmp_path / "split.cpp", tmp_path / "split"
    src.write_text(prog)
    subprocess.run(["g++", "-O1", "-std=c++17", "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert "cut 2" in r.stdout  # both part sizes occurred
