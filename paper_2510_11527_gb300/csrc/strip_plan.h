// Strip heights of the column-marching kernels (host code).
//
// Every warp marches S rows plus about 5 steps of warm-up and setup; CTAs of 4 warps are
// dealt to the SMs and R of them are resident. How long a step is depends on how many CTAs
// share the SM: t[r - 1] microseconds with r of them. A launch is estimated as its work at
// full residency plus `tail` times one strip's time alone: taller strips repeat less
// warm-up, but a strip along a front, where the limiter works, lasts past all others
// (degenerate Burgers 2048^2, per step: 0.44 ms with 16 to 26 rows, 0.48 with 32, 0.56 with
// 64 in one wave). The heavy kernels' strips are alike, so for them whole waves count (the
// busiest SM's CTAs, R at a time) more than the work (blended Buckley-Leverett 2048^2: 28
// rows, 3.0 waves, 1.14 ms; 26 rows 1.26 ms; 4096^2: 84 rows 3.87, 56 rows 4.03 ms), and
// for a batch's items as much (16 meshes, 5.6 million cells, one step: 29 rows 617, 23 rows
// 642 us). Against a fixed number of waves: Burgers 100^2 23 -> 12 us per stage, 512^2 128
// -> 85 us per step; Buckley-Leverett 1024^2 101 -> 54 us per stage (with its loop-free wave
// speeds).
//
// The light kernel on a single mesh (Burgers, linear flux) is the exception: the estimate is
// flat around its minimum there, and what counts is how the last wave ends (strip_rows_light).
#pragma once

namespace af {

struct StripPlan {
  int S;
  double cost;   // microseconds, relative for the heavy kernels
};

struct MarchKind {
  int R;
  double t[4];
  double waves, tail;   // weights of the waves (against the work) and of the tail
};
constexpr MarchKind MARCH_ZERO = {4, {1.05, 1.18, 1.40, 1.60}, 0.0, 1.0};    // one column per lane, zero flux
constexpr MarchKind MARCH_HEAVY = {3, {0.68, 0.82, 1.00, 0.0}, 0.7, 0.5};    // Buckley-Leverett, blends (relative)
constexpr MarchKind MARCH_ITEMS = {4, {1.12, 1.25, 1.50, 1.72}, 0.5, 0.5};   // a batch's items, dealt to one wave
constexpr MarchKind MARCH_PAIR = {3, {1.22, 1.40, 1.69, 0.0}, 0.0, 1.0};     // two columns per lane (zero flux)

// estimated time of w strips of S rows
inline double strip_cost(const MarchKind& k, int S, long long w) {
  const long long q = (w + 4 * 152 * 97 / 100) / (4 * 152);   // CTAs of the busiest SM, but for a few
  const int rest = (int)(q % k.R);
  const double waves = (double)(q / k.R) * k.t[k.R - 1] + (rest ? k.t[rest - 1] : 0.0);
  const double work = (double)w / (4 * 152) * k.t[k.R - 1] / k.R;
  return (S + 5) * (k.waves * waves + (1.0 - k.waves) * work + k.tail * k.t[0]);
}

// warps(S): how many warps strips of S rows make
template <class F>
inline StripPlan strip_plan(const MarchKind& k, F&& warps) {
  StripPlan best{4, -1.0};
  for (int S = 4; S <= 128; S += S < 32 ? 1 : 4) {
    const double cost = strip_cost(k, S, warps(S));
    if (best.cost < 0.0 || cost < best.cost) best = StripPlan{S, cost};
  }
  return best;
}

// Strip height of the light kernel on a single mesh of `bands` bands and ny rows: one and a
// quarter waves of 16 warps per SM as long as 4 to 16 rows give them, else two and a half of
// at most 48 rows. Both leave the SMs that are done early a short rest; full last waves, and
// those that end at a half between, wait for the strips along fronts. Degenerate Burgers, us
// per step on fresh discs / after 300 steps, as the estimate would choose and so: 512^2 85 /
// 92 and 79 / 88, 950^2 159 / 151 and 143 / 154, 1024^2 169 / 166 and 159 / 170, 1250^2 218 /
// 223 and 211 / 208, 300 x 4000 201 / 198 and 193 / 186, 2048^2 439 / 427 both, 3000^2 851 /
// 836 and 827 / 810, 4096^2 1471 / 1453 and 1481 / 1461 (with 100 rows, two and a half waves
// there, 1491 / 1463). Over 26 meshes from 200^2 to 4096^2 within 0.4 % of two and a half
// waves of 16 to 128 rows, the rule before, or faster, and within 3 % of the estimate.
inline int strip_rows_light(long long bands, int ny) {
  constexpr long long wave = 152 * 16;
  auto rows = [=](long long warps) { return (bands * ny + warps - 1) / warps; };
  const long long one = rows(wave * 5 / 4), two = rows(wave * 5 / 2);
  if (one <= 16) return one < 4 ? 4 : (int)one;
  return two > 48 ? 48 : (int)two;
}

}  // namespace af
