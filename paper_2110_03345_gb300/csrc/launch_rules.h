// Rules that choose between kernels and launch shapes from sizes alone (host code without
// CUDA types, so that they can be checked without a GPU).
#pragma once

namespace fwi {

// Whether a 3D call makes and uses the density flags (launch_density_flags): `points` grid
// points in all slots, nt time samples.  Making them costs 40 us on a small grid, 90 at 192
// x 180 x 200, 160 at 256^3 and 320-430 at 384^3.  Small launches are bound by latency, not
// by the loads and the arithmetic that the flags spare, and lose to the choice per plane.
// Gain per step (step pair for gradients) with a density that is constant within two
// tissues, order 10, in us: leapfrog forward 100^3 -0.4, 128^3 -0.2, 152 x 160 x 176 0, 192
// x 180 x 200 2.5, 256^3 8.4, 384^3 53; gradient -1.8, -1.3, -0.4, 11.8, 20.6, 118; PML
// forward 64^3 0, 100^3 0.6, 300 x 64 x 64 2.2, 128^3 4.2, 256^3 17; gradient 0, 2.3, 5.8, 5.9,
// 56.  So the leapfrog takes them from 5.5 million points, the PML from a million, and
// either where the run is long enough to win their cost back (8-37 steps).
inline bool density_flags_pay(long long points, int nt, bool grad, bool pml) {
  return points >= (pml ? 1000000LL : 5500000LL) && (grad ? 4LL : 1LL) * nt >= 40;
}

}  // namespace fwi
