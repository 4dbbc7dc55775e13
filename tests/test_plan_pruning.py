"""The tile plans skip candidates that cannot win; they must name the same plan as the
model evaluated over every candidate (compiled with nvcc and run on the CPU, no GPU)."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2005_08674_gb300", "csrc")

DRIVER = r"""
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include "lbm_multistep.cuh"
using namespace lbmk;

// the models of plan_tiles and plan_resident, over every candidate
static TilePlan all_tiles(int nx, int ny, bool f64, bool px, bool py, int sms) {
  // microseconds, measured: launch, load per node, step, node, boundary node
  const double t_launch = 2.0, t_load = f64 ? 1.4e-3 : 0.7e-3, t_step = f64 ? 0.9 : 0.35;
  const double t_node = f64 ? 15e-3 : 0.45e-3, t_edge = f64 ? 100e-3 : 3e-3;
  const size_t elt = f64 ? 8 : 4, room = kTileRoom;
  TilePlan best;
  for (int steps : {1, 2, 3, 4, 5, 6, 8, 10, 12})
    for (int gx = 1; gx <= 64 && nx / gx >= 4; ++gx)
      for (int gy = 1; gy <= 64 && ny / gy >= 4; ++gy) {
        if (gx * gy > 8 * sms) break;
        const int tw = (nx + gx - 1) / gx, th = (ny + gy - 1) / gy;
        const int w = px || gx > 2 ? tw + 2 * steps : (gx == 2 ? tw + steps : tw);
        const int h = py || gy > 2 ? th + 2 * steps : (gy == 2 ? th + steps : th);
        if ((px && w > nx) || (py && h > ny)) continue;
        const size_t smem = 2 * 9 * (size_t)w * h * elt;
        if (smem > room) continue;
        const int waves = (gx * gy + sms - 1) / sms;
        double block = 0.8 + t_load * w * h;
        for (int j = 1; j <= steps; ++j) {
          const double c = (double)(steps - j) / steps;  // of the halo that step j still covers
          const double wj = tw + (w - tw) * c, hj = th + (h - th) * c;
          block += t_step + t_node * wj * hj + t_edge * std::max(wj, hj);
        }
        const double us = (t_launch + waves * block) / steps;
        if (us < best.us) best = TilePlan{gx, gy, steps, (int)smem, us};
      }
  return best;
}

static TilePlan all_resident(int nx, int ny, bool px, bool py, int sms) {
  // microseconds: a round's exchange, halo node, step (the boundary's chain of operations), row of 64 nodes,
  // boundary node (of a corner tile; both lines of a periodic axis)
  const double t_round = 2.6, t_halo = 0.7e-3, t_step = 0.9, t_row = 0.025, t_edge = 0.01;
  TilePlan best;
  for (int halo = 1; halo <= 8; ++halo) {
    const int side = std::max(4, halo);  // a halo reaches no further than the next tile
    for (int gx = 1; gx <= sms && nx / gx >= side; ++gx)
      for (int gy = 1; gx * gy <= sms && ny / gy >= side; ++gy) {
        const int tw = (nx + gx - 1) / gx, th = (ny + gy - 1) / gy;
        const int w = px || gx > 2 ? tw + 2 * halo : (gx == 2 ? tw + halo : tw);
        const int h = py || gy > 2 ? th + 2 * halo : (gy == 2 ? th + halo : th);
        if ((px && w > nx) || (py && h > ny)) continue;
        const size_t smem = tile_bytes<float>(w, h) + kRowSlack * sizeof(float);
        if (smem > kTileRoom) continue;
        double us = t_round + t_halo * ((double)w * h - (double)tw * th);
        for (int j = 1; j <= halo; ++j) {
          const double c = (double)(halo - j) / halo;  // of the halo that step j still covers
          const double wj = tw + (w - tw) * c, hj = th + (h - th) * c;
          const double edge = (px || gx == 1 ? 2 : 1) * hj + (py || gy == 1 ? 2 : 1) * wj;
          us += t_step + t_row * (int)((wj + 63) / 64) * hj + t_edge * edge;
        }
        if (us / halo < best.us) best = TilePlan{gx, gy, halo, (int)smem, us / halo};
      }
  }
  return best;
}

static bool same(const TilePlan& a, const TilePlan& b) {
  return a.gx == b.gx && a.gy == b.gy && a.steps == b.steps && a.smem == b.smem;
}

int main() {
  std::mt19937 r(1);
  std::uniform_real_distribution<> side(0, 9);
  int plans = 0, differ = 0;
  while (plans < 1500) {
    const int nx = 8 + (int)std::exp(side(r)), ny = 8 + (int)std::exp(side(r));
    if ((long long)nx * ny > 1 << 21) continue;
    const bool f64 = r() & 1, px = (r() & 3) == 0, py = (r() & 3) == 0;
    ++plans;
    if (same(all_tiles(nx, ny, f64, px, py, 152), plan_tiles(nx, ny, f64, px, py, 152)) &&
        same(all_resident(nx, ny, px, py, 152), plan_resident(nx, ny, px, py, 152)))
      continue;
    ++differ;
    std::printf("%d x %d f64 %d periodic %d %d\n", nx, ny, f64, px, py);
  }
  std::printf("%d differ\n", differ);
  return differ != 0;
}
"""


def test_pruned_plans_are_the_best(tmp_path):
    from paper_2005_08674_gb300 import build
    src, exe = tmp_path / "plan.cu", tmp_path / "plan"
    src.write_text(DRIVER)
    r = subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I", CSRC, "-I",
                        build.INCLUDE, str(src), "-o", str(exe)], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
