"""Host side of the resident tiles, compiled with nvcc and run on the CPU (no GPU
needed): the tiles cover the domain once, fit a block's shared memory, and every
element of a tile's halo is named once and belongs to one of the eight
neighbours, among the nodes that neighbour writes out."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2005_08674_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include <vector>
#include "lbm_multistep.cuh"
using namespace lbmk;

static int check(int nx, int ny, bool px, bool py, int sms) {
  const TilePlan p = plan_resident(nx, ny, px, py, sms);
  if (p.steps == 0) return 0;
  const int H = p.steps;
  if (p.gx * p.gy > sms) return 1;
  auto tile = [&](int tx, int ty) {
    return TileRect{nx * tx / p.gx, ny * ty / p.gy, nx * (tx + 1) / p.gx, ny * (ty + 1) / p.gy};
  };
  std::vector<int> owner((size_t)nx * ny, -1);
  for (int k = 0; k < p.gx * p.gy; ++k) {
    const TileRect t = tile(k % p.gx, k / p.gx);
    for (int y = t.y0; y < t.y1; ++y)
      for (int x = t.x0; x < t.x1; ++x) {
        if (owner[(size_t)y * nx + x] != -1) return 2;
        owner[(size_t)y * nx + x] = k;
      }
  }
  for (int v : owner)
    if (v < 0) return 3;
  for (int k = 0; k < p.gx * p.gy; ++k) {
    const int tx = k % p.gx, ty = k / p.gx;
    const TileRect t = tile(tx, ty);
    const TileRegion reg = tile_region(nx, ny, px, py, t, H);
    // rows are read up to 64 nodes and one past their ends
    if (tile_bytes<float>(reg.w, reg.h) + 65 * sizeof(float) > (size_t)p.smem || (size_t)p.smem > kTileRoom) return 4;
    if (9ull * reg.w * reg.h * reg.w >= 1ull << 32) return 5;
    std::vector<int> seen((size_t)9 * reg.w * reg.h, 0);
    const TileHalo h(t, reg);
    for (int e = 0; e < h.n; ++e) {
      int i, lx, ly;
      h.at(e, i, lx, ly);
      if (i < 0 || i > 8 || lx < 0 || lx >= reg.w || ly < 0 || ly >= reg.h) return 6;
      int x = reg.x0 + lx, y = reg.y0 + ly;
      if (x >= t.x0 && x < t.x1 && y >= t.y0 && y < t.y1) return 7;  // the tile's own
      if (seen[(9 * ly + i) * reg.w + lx]++) return 8;
      x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
      y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
      if (x < 0 || x >= nx || y < 0 || y >= ny) return 9;
      const int o = owner[(size_t)y * nx + x], ox = o % p.gx, oy = o / p.gx;
      auto near = [](int a, int b, int n, bool wrap) {
        const int d = a > b ? a - b : b - a;
        return d <= 1 || (wrap && d == n - 1);
      };
      if (!near(ox, tx, p.gx, px) || !near(oy, ty, p.gy, py)) return 10;
      const TileRect u = tile(ox, oy);  // written out by its owner: outside the owner's core
      const int cx0 = px || u.x0 > 0 ? u.x0 + H : u.x0, cx1 = px || u.x1 < nx ? u.x1 - H : u.x1;
      const int cy0 = py || u.y0 > 0 ? u.y0 + H : u.y0, cy1 = py || u.y1 < ny ? u.y1 - H : u.y1;
      if (x >= cx0 && x < cx1 && y >= cy0 && y < cy1) return 11;
    }
    // the boundary's slots: every perimeter node of the widest rectangle once
    const EdgeList list(t, H - 1, nx, ny, px, py);
    std::vector<int> edge((size_t)reg.w * reg.h, 0);
    for (int k = 0; k < list.n; ++k) {
      int x, y;
      if (!list.node(k, nx, ny, x, y)) continue;
      if (x < reg.x0 || x >= reg.x0 + reg.w || y < reg.y0 || y >= reg.y0 + reg.h) return 13;
      ++edge[(size_t)(y - reg.y0) * reg.w + x - reg.x0];
    }
    for (int y = list.ay; y < list.by; ++y)
      for (int x = list.ax; x < list.bx; ++x) {
        const bool per = x == 0 || x == nx - 1 || y == 0 || y == ny - 1 || x == -1 || x == nx || y == -1 || y == ny;
        if (edge[(size_t)(y - reg.y0) * reg.w + x - reg.x0] != (per ? 1 : 0)) return 14;
      }
    long long covered = 0;
    for (int v : seen) covered += v;
    if (covered != 9LL * (reg.w * reg.h - (t.x1 - t.x0) * (t.y1 - t.y0))) return 12;
  }
  return 0;
}

int main() {
  for (int nx : {8, 9, 13, 64, 100, 131, 200, 257, 401, 613})
    for (int ny : {8, 11, 40, 128, 200, 377, 640})
      for (int m = 0; m < 4; ++m)
        for (int sms : {152, 148, 7})
          if (int rc = check(nx, ny, m & 1, m & 2, sms)) {
            printf("%d %d %d %d: %d\n", nx, ny, m, sms, rc);
            return rc;
          }
  printf("ok\n");
  return 0;
}
"""


def test_resident_plan(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "plan.cu", tmp_path / "plan"
    src.write_text(DRIVER)
    subprocess.check_call([nvcc, "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-arch=sm_103a", "-I", CSRC,
                           "-o", str(exe), str(src)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
