"""The z-marching 3D stage's choice of strips (host code, compiled with the host compiler):
the cheapest height, as trying every number of strips finds it, without that many trials."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <chrono>
#include <cstdio>
#include <initializer_list>
#include "march3d_plan.h"
static af::M3Plan every(const int* n, int TY) {
  af::M3Plan p;
  p.bands = (n[0] + af::M3_BAND - 1) / af::M3_BAND;
  p.rows = (n[1] + TY - 5) / (TY - 4);
  p.S = n[2];
  const long long tiles = (long long)p.bands * p.rows;
  double best = -1.0;
  for (int s = 1; s <= n[2] && s <= 152 * 8; ++s) {
    const int L = (n[2] + s - 1) / s;
    const long long waves = (tiles * ((n[2] + L - 1) / L) + 151) / 152;
    if (best < 0.0 || waves * (L + 1.2) < best) {
      best = waves * (L + 1.2);
      p.S = L;
    }
  }
  p.cost = best * (TY - 4 + 0.8) * (TY > af::M3_ROWS_SMALL ? 3.0 : 3.4);
  return p;
}
template <class F>
static double seconds(F plan) {
  volatile int sink = 0;
  const auto t0 = std::chrono::steady_clock::now();
  for (int k = 0; k < 2000; ++k) {
    const int n[3] = {20 + k % 3, 8, 1216};
    sink = sink + plan(n, 12).S;
  }
  return std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
}
int main() {
  for (int nz = 1; nz <= 2600; nz += nz < 400 ? 1 : 37)
    for (int nx : {1, 28, 29, 300})
      for (int ny : {1, 8, 81, 500})
        for (int TY : {8, 12, 16}) {
          const int n[3] = {nx, ny, nz};
          const af::M3Plan a = af::m3_plan(n, TY), b = every(n, TY);
          if (a.S != b.S || a.cost != b.cost || a.bands != b.bands || a.rows != b.rows) {
            std::printf("%d %d %d rows %d: %d / %d\n", nx, ny, nz, TY, a.S, b.S);
            return 1;
          }
        }
  const double a = seconds(af::m3_plan), b = seconds(every);
  std::printf("%.3g %.3g\n", a, b);
  return 4 * a < b ? 0 : 2;
}
"""


def test_same_choice_as_trying_every_number_of_strips(tmp_path):
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2510_11527_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
