"""The exchange relation of the heat kernel's resident tiles (csrc/heat_geom.h, the
functions heat_tile.cu itself runs), enumerated on the CPU: a block may overwrite the
words of an exchange two exchanges later only because every block that reads them is one
it waits for itself.  So "waits for" has to be symmetric whatever the obstacles are, and
every awaited cell has to be one its owner sends."""
import shutil
import subprocess

import numpy as np
import pytest

PROGRAM = r"""
#include <cstdio>
#include <set>
#include <utility>
#include <vector>
#include "heat_geom.h"
using namespace jko::heat_geom;
int main(int, char** a) {
  int nx, ny, sms;
  FILE* f = std::fopen(a[1], "r");
  if (std::fscanf(f, "%d %d %d", &nx, &ny, &sms) != 3) return 1;
  std::vector<uint8_t> m((size_t)nx * ny);
  for (auto& v : m) { int b; if (std::fscanf(f, "%d", &b) != 1) return 1; v = (uint8_t)b; }
  int tw = 0, th = 0;
  tile_shape(nx, ny, sms, &tw, &th);
  const int ntx = (nx + tw - 1) / tw, nb = ntx * ((ny + th - 1) / th);
  std::set<std::pair<int, int>> waits;
  int unsent = 0, outside = 0;
  for (int b = 0; b < nb; ++b) {
    const Tile t = tile_of(b, tw, th, ntx, nx, ny);
    const float inv = 1.0f / (float)(t.w + 2 * H);
    std::set<std::pair<int, int>> seen;
    for (int i = 0; i < ring_cells(t); ++i) {
      int ex, ey;
      ring_place(i, t, inv, ex, ey);
      if (!seen.insert({ex, ey}).second || (ex >= H && ex < H + t.w && ey >= H && ey < H + t.h) ||
          ex < 0 || ey < 0 || ex >= t.w + 2 * H || ey >= t.h + 2 * H) ++outside;
      const int x = t.x0 + ex - H, y = t.y0 + ey - H;
      const int fl = cell_flags(x, y, nx, ny, m.data());
      if (!awaited(fl)) continue;
      const int o = y / th * ntx + x / tw;
      const Tile ot = tile_of(o, tw, th, ntx, nx, ny);
      if (!sent(x - ot.x0, y - ot.y0, ot)) ++unsent;
      waits.insert({b, o});
    }
  }
  int one_way = 0;
  for (auto& p : waits) one_way += !waits.count({p.second, p.first});
  std::printf("%d %d %d %d %d %d %d\n", nb, (int)waits.size(), one_way, unsent, outside,
              (int)tile_bytes(tw, th, 4), (int)tile_bytes(tw, th, 8));
}
"""


@pytest.fixture(scope="module")
def relation(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    import os
    import paper_1502_06216_gb300
    csrc = os.path.join(os.path.dirname(paper_1502_06216_gb300.__file__), "csrc")
    d = tmp_path_factory.mktemp("tiles")
    (d / "p.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", csrc, str(d / "p.cpp"), "-o", str(d / "p")],
                   check=True)

    def run(nx, ny, sms, mask):
        (d / "in").write_text(f"{nx} {ny} {sms}\n" + " ".join(map(str, mask.astype(int).ravel())))
        out = subprocess.run([str(d / "p"), str(d / "in")], check=True, capture_output=True, text=True)
        return tuple(map(int, out.stdout.split()))
    return run


def obstacles(nx, ny):
    X, Y = np.meshgrid((np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny)
    yield "none", np.zeros((ny, nx), bool)
    yield "two rooms", (np.abs(X - 0.5) < 0.02) & (np.abs(Y - 0.5) >= 0.1)
    yield "thick wall", (np.abs(X - 0.5) < 0.12) & (np.abs(Y - 0.5) >= 0.1)
    yield "closed wall", np.abs(Y - 0.4) < 0.1
    yield "disk", (X - 0.5) ** 2 + (Y - 0.5) ** 2 < 0.04
    yield "square", (np.abs(X - 0.45) < 0.15) & (np.abs(Y - 0.45) < 0.15)


@pytest.mark.parametrize("nx,ny", [(30, 20), (96, 90), (100, 100), (150, 150), (200, 200), (48, 40),
                                   (37, 61), (1, 64), (64, 1), (5, 4)])
def test_waiting_is_symmetric_and_awaited_cells_are_sent(relation, nx, ny):
    for sms in (148, 152):
        for name, mask in obstacles(nx, ny):
            blocks, waits, one_way, unsent, outside, _, _ = relation(nx, ny, sms, mask)
            print(nx, ny, sms, name, blocks, waits, one_way, unsent, outside)
            assert blocks <= sms
            assert one_way == 0, name
            assert unsent == 0, name
            assert outside == 0, name


def test_grids_beyond_the_tiles(relation):
    """The sizes at which heat.cu's persistent kernel (several tiles a block) still runs, as
    the GPU test of that kernel takes them: the tile does not fit the 227 KB of a block."""
    smem = 227 * 1024
    for sms in (148, 152):
        fits = lambda n, m: relation(n, m, sms, np.zeros((m, n), bool))[5:]
        assert fits(900, 880)[0] > smem and fits(760, 800)[1] > smem
        assert fits(840, 840)[0] <= smem and fits(700, 700)[1] <= smem
