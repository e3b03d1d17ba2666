// Rules that choose between kernels and launch shapes from sizes alone (host code without
// CUDA types, so that they can be checked without a GPU).
#pragma once

#include <cmath>

namespace fwi {

// Whether a 3D call makes and uses the density flags (launch_density_flags): `points` grid
// points in all slots, nt time samples.  Making them costs 40 us on a small grid, 90 at 192
// x 180 x 200, 160 at 256^3 and 320-430 at 384^3.  Small launches are bound by latency, not
// by the loads and the arithmetic that the flags spare, and lose to the choice per plane.
// Gain per step (step pair for gradients) with a density that is constant within two
// tissues, order 10, in us: leapfrog forward 100^3 -0.4, 128^3 -0.2, 150^3 -0.2, 152 x 160 x
// 176 0, 130 x 226 x 143 3, 192 x 180 x 200 2.5, 256^3 8.4, 384^3 53; gradient -1.8, -1.3, 2.6,
// -0.4, 12, 11.8, 20.6, 118, four shots of 300 x 64 x 64 6.7; PML forward 64^3 0, 100^3 0.6,
// 300 x 64 x 64 2.2, 128^3 4.2, 256^3 17; gradient 0, 2.3, 5.8, 5.9, 56.  So the leapfrog takes
// them from three million points, the PML from a million, and either where the run is long
// enough to win their cost back.
inline bool density_flags_pay(long long points, int nt, bool grad, bool pml) {
  return points >= (pml ? 1000000LL : 3000000LL) &&
         (grad ? 4LL : 1LL) * nt >= (points >= 6000000LL ? 40 : pml ? 60 : 160);
}

// Planes per CTA of the default 3D variant (0: none fits `most_chunks`), for `cols` column
// tiles over all slots.  A CTA of zc planes spends about zc + 5 plane times (the 2R halo
// planes before its first point cost less than computed ones; PML zc + 3, two of its passes
// have none or few); three share an SM, two in the variable-density adjoint and the PML.
// With x CTAs per place a launch takes between ceil(x) of these, if all keep step, and x + a
// tail, if they drift apart: a weighted mean of the two.
// (Rounds alone, the rule before this one, took a half-empty round of 48 planes at 192
// planes and 1.84 rounds of 46 at 320.)
// us per step / step pair, order 10, one shot, 32 planes -> rounds alone -> this rule.  With
// density: 128^3 45.6 -> 18.8 -> 18.8 / 94.2 -> 51.2 -> 51.2, 152 x 160 x 176 51.4 -> 38.4 -> 38.4 /
// 103.2 in all, 192 x 180 x 200 68.7 -> 75.8 -> 63.8 / 161.0 -> 158.9 -> 158.9, 256^3 115.7 ->
// 108.5 -> 108.5 / 282.6 -> 264.1 -> 264.1.  Without: 192 x 180 x 200 67.1 -> 64.5 -> 54.6 / 152.5 ->
// 142.3 -> 122.1, 96 x 300 x 300 69.3 -> 64.4 -> 57.8 / 157.3 -> 144.1 -> 130.2, 320 x 240 x 200
// 110.6 -> 116.0 -> 107.4 / 250.2 -> 259.1 -> 242.3.  PML: 192 x 180 x 200 257.4 -> 303.4 -> 213.0 /
// 537.0 -> 486.6 -> 483.1, 256^3 365.3 -> 363.8 -> 342.3 / 833.7 -> 821.7 -> 803.7.
inline int z_planes(int nsm, int nz, long long cols, bool vd, bool grad, bool pml, int most_planes,
                    long long most_chunks) {
  int best = 0;
  double least = 0.0;
  for (int nzc = 1; nzc <= nz && nzc <= most_chunks; ++nzc) {
    const int zc = (nz + nzc - 1) / nzc;
    if (zc > most_planes || (nz + zc - 1) / zc != nzc) continue;
    if (zc < 8 && best > 0) break;
    auto cost = [&](int per_sm, int halo, double rounds, double tail) {
      const double x = (double)(cols * nzc) / ((double)per_sm * nsm);
      return (zc + halo) * (rounds * std::ceil(x) + (1.0 - rounds) * (x + tail));
    };
    const double fwd = cost(3, 5, 0.8, 1.3), adj = vd ? cost(2, 5, 0.9, 1.3) : fwd;
    const double c = pml ? cost(2, 3, 0.6, 1.6) : fwd + (grad ? adj : 0.0);
    if (best == 0 || c < least) {
      best = zc;
      least = c;
    }
  }
  return best;
}

// Whether runs of `nt` samples (gradients: between checkpoints every K steps, 0: none) are
// long enough for resident launches.  A launch loads and stores the whole state and a call
// clears the exchange buffer, some 20 us each.  One shot with density on 256 x 256, 456 x
// 485, 700 x 748 and 1024 x 1024, times summed, per-step -> resident: gradient of 200 steps
// with K = 1 32.1 -> 53.0 ms, 2 22.8 -> 28.9, 4 17.5 -> 18.1, 6 16.1 -> 14.6 (700 x 748 alone 3.9 ->
// 4.2), 8 15.2 -> 12.7; forward of nt - 1 = 1 747 -> 825 us, 4 802 -> 850, 8 882 -> 890, 16 1020 ->
// 968; gradient of 2 1032 -> 1111, 8 1315 -> 1256.
inline bool resident_run(int nt, int K, bool grad) {
  return grad && K > 0 && K < nt - 1 ? K >= 6 : nt - 1 >= (grad ? 8 : 12);
}

// Whether a resident call beats the per-step kernels: `units` is choose_res's estimate of a
// resident step (all rounds of shots), `shot_times` shot_group's of a per-step launch.  The
// estimates in us are fits over nine grids of 256 x 256 - 1024 x 1024 and one to 32 shots
// (8th order; residuals 8%); within 2% of each other the call stays resident.  Without this
// a last round of few shots was not seen (resident / per-step, us per step or step pair):
// 456 x 485 with density, forward of 8, 9 and 10 shots 8.6 / 9.4, 10.5 / 10.2, 12.2 / 10.2; gradient
// of 12 and 13 shots 30.1 / 31.3, 39.5 / 31.4; 700 x 748 gradient of 6 and 7 29.3 / 32.2, 38.6 / 35.0.
inline bool resident_pays(double units, double shot_times, bool grad, bool vd) {
  const double per_step = grad ? (vd ? 4.23 + 3.13 * shot_times : 4.25 + 2.38 * shot_times)
                               : (vd ? 2.50 + 1.12 * shot_times : 2.73 + 0.89 * shot_times);
  const double resident = units * (grad ? (vd ? 0.0546 : 0.0418) : (vd ? 0.0234 : 0.0193));
  return resident <= 1.02 * per_step;
}

}  // namespace fwi
