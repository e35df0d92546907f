"""Strip heights of the light column-marching kernel (host code, compiled with the host
compiler): one and a quarter waves of warps as long as 4 to 16 rows give them, else two and
a half of at most 48 rows."""
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
      const int S = af::strip_rows_light(bands, ny);
      const double waves = (double)bands * ny / S / (152 * 16), shorter = (double)bands * ny / (S - 1) / (152 * 16);
      const double want = (double)bands * ny / 16 / (152 * 16) <= 1.25 ? 1.25 : 2.5;
      // the shortest strips that make no more waves than wanted
      bool ok = S >= 4 && S <= 48 && (waves <= want || S == 48) && (shorter > want || S == 4);
      if (!ok) {
        std::printf("%d x %d: %d rows, %.2f waves\n", nx, ny, S, waves);
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
