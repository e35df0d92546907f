// Strip heights of the column-marching kernels (host code).
//
// Every warp marches S rows plus about 5 steps of warm-up and setup; CTAs of 4 warps are
// dealt to the SMs and R of them are resident. How long a step is depends on how many CTAs
// share the SM: t[r - 1] microseconds with r of them. Two estimates of a launch are
// averaged: its work at full residency, and its waves (the busiest SM's CTAs, R at a time),
// because CTAs are equal on smooth data and uneven where the limiter works. To that comes
// the tail, half of one strip's time on its own: fewer, taller strips repeat less warm-up
// but one strip along a front then lasts past all others (degenerate Burgers 2048^2, per
// step: 0.44 ms with 16 to 32 rows, 0.54 with 64 in one wave). Measured per stage against
// the fixed number of waves used before, smooth data: Burgers 100^2 23 -> 11 us, 1200^2
// 58 -> 45 us, Buckley-Leverett 1024^2 101 -> 54 us (with its loop-free wave speeds).
#pragma once

namespace af {

struct StripPlan {
  int S;
  double cost;   // microseconds, relative for the heavy kernels
};

struct MarchKind {
  int R;
  double t[4];
};
constexpr MarchKind MARCH_LIGHT = {4, {1.12, 1.25, 1.50, 1.72}};   // one column per lane
constexpr MarchKind MARCH_ZERO = {4, {1.05, 1.18, 1.40, 1.60}};    // the same, zero flux
constexpr MarchKind MARCH_HEAVY = {3, {0.68, 0.82, 1.00, 0.0}};    // Buckley-Leverett, blends (relative)
constexpr MarchKind MARCH_PAIR = {3, {1.22, 1.40, 1.69, 0.0}};     // two columns per lane (zero flux)

// warps(S): how many warps strips of S rows make
template <class F>
inline StripPlan strip_plan(const MarchKind& k, F&& warps) {
  StripPlan best{4, -1.0};
  for (int S = 4; S <= 128; S += S < 32 ? 1 : 4) {
    const long long w = warps(S), q = (w + 4 * 152 - 1) / (4 * 152);   // q: CTAs of the busiest SM
    const int rest = (int)(q % k.R);
    const double waves = (double)(q / k.R) * k.t[k.R - 1] + (rest ? k.t[rest - 1] : 0.0);
    const double work = (double)w / (4 * 152) * k.t[k.R - 1] / k.R;
    const double cost = (S + 5) * (0.5 * (waves + work) + 0.5 * k.t[0]);
    if (best.cost < 0.0 || cost < best.cost) best = StripPlan{S, cost};
  }
  return best;
}

}  // namespace af
