"""Strip heights of the light column-marching kernel (host code, compiled with the host
compiler): the estimate's choice where it predicts at least 5 % less than two and a half
waves of 16 to 48 rows, else these."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include <initializer_list>
#include "strip_plan.h"
int main() {
  for (int nx : {28, 100, 300, 512, 850, 1024, 1300, 2048, 3000, 4096, 20000})
    for (int ny : {1, 4, 100, 300, 512, 850, 1024, 1300, 2048, 3000, 4096, 20000}) {
      const long long bands = (nx + 27) / 28;
      const auto warps = [&](int S) { return bands * ((ny + S - 1) / S); };
      const af::StripPlan p = af::strip_plan_light(bands, ny), best = af::strip_plan(af::MARCH_LIGHT, warps);
      const double cost = af::strip_cost(af::MARCH_LIGHT, p.S, warps(p.S));
      bool ok = p.S >= 4 && p.S <= 128 && p.cost == cost && best.cost >= 0.95 * p.cost - 1e-9;
      if (p.S != best.S) {   // two and a half waves of 16 warps per SM, as far as 16 to 48 rows give them
        const double waves = (double)bands * ny / p.S / (152 * 16);
        ok = ok && p.S >= 16 && p.S <= 48 && (p.S == 48 || waves <= 2.5) && (p.S == 16 || waves >= 2.3);
      }
      if (!ok) {
        std::printf("%d x %d: %d rows (estimate's choice %d)\n", nx, ny, p.S, best.S);
        return 1;
      }
    }
  return 0;
}
"""


def test_strip_heights_of_the_light_march(tmp_path):
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2510_11527_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
