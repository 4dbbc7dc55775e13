"""Host side of the multi-step forms, compiled with nvcc and run on the CPU (no
GPU needed): the frame tiles and the rolling part cover every node of a domain
exactly once for every number of steps, frame tiles fit the shared memory of
their blocks, and a small domain's tiles cover it, fit a block's shared memory
and are never thinner than the boundary's difference needs."""
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

static int frame(int nx, int ny, int D) {
  std::vector<int> seen((size_t)nx * ny, 0);
  for (int k = 0; k < frame_tiles(nx, ny); ++k) {
    const TileRect t = frame_tile(nx, ny, D, k);
    if (t.y0 >= t.y1) continue;
    if (t.x0 < 0 || t.y0 < 0 || t.x1 > nx || t.y1 > ny || t.x0 >= t.x1) return 1;
    const int w = std::min(t.x1 + D, nx) - std::max(t.x0 - D, 0), h = std::min(t.y1 + D, ny) - std::max(t.y0 - D, 0);
    if (tile_bytes<float>(w, h) > Roll<float>::kSmem || tile_bytes<float>(w, h) > Roll<__half>::kSmem) return 2;
    if ((t.x0 == 0 || t.x1 == nx) && t.x1 - t.x0 < 2) return 3;
    if ((t.y0 == 0 || t.y1 == ny) && t.y1 - t.y0 < 2) return 4;
    for (int y = t.y0; y < t.y1; ++y)
      for (int x = t.x0; x < t.x1; ++x) ++seen[(size_t)y * nx + x];
  }
  for (int y = 0; y < ny; ++y)
    for (int x = 0; x < nx; ++x) {
      const bool rolled = x >= D && x < nx - D && y >= D && y < ny - D;
      if (seen[(size_t)y * nx + x] != (rolled ? 0 : 1)) return 5;
    }
  // strips: output columns X0 + D .. X0 + D + OUT, inside the columns that
  // are valid after D steps, and starting on 16 bytes
  for (int out : {Roll<float>::OUT, Roll<__half>::OUT})
    if (out + 2 * D > Roll<float>::W) return 6;
  if (Roll<float>::OUT * 4 % 16 || Roll<__half>::OUT * 2 % 16) return 7;
  return 0;
}

static int tiles(int nx, int ny, bool f64, bool px, bool py) {
  const TilePlan p = plan_tiles(nx, ny, f64, px, py, 152);
  if (p.steps == 0) return px || py ? 0 : 10;  // (a periodic axis may be too short to cut)
  const int D = p.steps;
  std::vector<int> seen((size_t)nx * ny, 0);
  for (int ty = 0; ty < p.gy; ++ty)
    for (int tx = 0; tx < p.gx; ++tx) {
      const int x0 = nx * tx / p.gx, x1 = nx * (tx + 1) / p.gx, y0 = ny * ty / p.gy, y1 = ny * (ty + 1) / p.gy;
      const int w = px ? x1 - x0 + 2 * D : std::min(x1 + D, nx) - std::max(x0 - D, 0);
      const int h = py ? y1 - y0 + 2 * D : std::min(y1 + D, ny) - std::max(y0 - D, 0);
      if (2ull * 9 * w * h * (f64 ? 8 : 4) > (unsigned long long)p.smem || (size_t)p.smem > kTileRoom) return 11;
      if ((px && w > nx) || (py && h > ny)) return 12;
      if (x1 - x0 < 2 || y1 - y0 < 2) return 13;
      for (int y = y0; y < y1; ++y)
        for (int x = x0; x < x1; ++x) ++seen[(size_t)y * nx + x];
    }
  for (int v : seen)
    if (v != 1) return 14;
  return 0;
}

int main() {
  for (int nx : {8, 9, 15, 40, 41, 63, 64, 65, 119, 300, 517})
    for (int ny : {8, 9, 10, 12, 17, 43, 44, 45, 84, 85, 301})
      for (int D = 2; D <= kPassSteps; ++D)
        if (int rc = frame(nx, ny, D)) { printf("frame %d %d %d: %d\n", nx, ny, D, rc); return rc; }
  for (int nx : {8, 9, 13, 64, 100, 131, 200, 257, 401})
    for (int ny : {8, 11, 40, 128, 200, 333})
      for (int m = 0; m < 8; ++m)
        if (int rc = tiles(nx, ny, m & 1, m & 2, m & 4)) { printf("tiles %d %d %d: %d\n", nx, ny, m, rc); return rc; }
  printf("ok\n");
  return 0;
}
"""


def test_plans_cover_every_node_once(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "plan.cu", tmp_path / "plan"
    src.write_text(DRIVER)
    subprocess.check_call([nvcc, "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-arch=sm_103a", "-I", CSRC,
                           "-o", str(exe), str(src)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
