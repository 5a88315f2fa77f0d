// olb_fold.h -- host-side constants of the FP64 collision (collide_folded).
#pragma once

#include <cmath>

namespace olb {

// Constants of the FP64 collision, formed once on the host: on this GPU an FP64
// instruction of a warp holds an SM's FP64 pipe for 16 cycles, so products of uniform
// values are not left to the threads.  Weight classes 0: rest, 1, 2: the moving
// velocities (along an axis, diagonal).
struct Fold64 {
  double keep, even, odd;      // 1 - omega, (1 - omega)/2 and (1 - omega_odd)/2
  double ow[3], b[3], t[3];    // omega w, 4.5 omega w, 3 omega_odd w
  double gu[3];                // 3 (1 - omega/2) w
  double gq[9], ga[9];         // 9 (1 - omega/2) w_k c_k.F,  3 (1 - omega_odd/2) w_k c_k.F
};

// The constants without a force (dim 2: D2Q9, 3: D3Q19).
//
// A step multiplies the mass by keep + ow[0] + n1 ow[1] + n2 ow[2] and the momentum by
// 2 odd + 2 t[1] + m t[2] (n1, n2: moving velocities of each class, m = 4 in 2D, 8 in
// 3D), both 1 in exact arithmetic.  Products rounded one by one leave factors of up to
// 1 - 2.2e-16, the same at every step and in every cell: a drift that grows with the
// number of steps (64^2 vortex, tau = 0.8, 500 steps: error 5.4e-14 against 2.7e-14 of
// the unfolded collision).  So ow[0] and t[1] are formed as remainders, and the others
// are rounded to multiples of a quantum (at most 4 of their own units in the last place)
// that makes the remainders exact: both factors are 1 with no rounding.
inline Fold64 fold64_rates(int dim, double omega, double omega_odd) {
  const bool flat = dim == 2;
  const double w[3] = {flat ? 4.0 / 9.0 : 1.0 / 3.0, flat ? 1.0 / 9.0 : 1.0 / 18.0, 1.0 / 36.0};
  const double n1 = flat ? 4.0 : 6.0, n2 = flat ? 4.0 : 12.0, m = flat ? 4.0 : 8.0;
  // unit in the last place of x (of the next larger binade just below a power of two,
  // where the remainder may round up into it)
  auto ulp = [](double x) { return std::ldexp(1.0, std::ilogb(x * (1.0 + 1e-12)) - 52); };
  auto multiple = [](double x, double q) { return std::rint(x / q) * q; };
  Fold64 r = {};
  r.keep = 1.0 - omega;
  r.even = 0.5 * r.keep;
  r.odd = 0.5 * (1.0 - omega_odd);
  for (int c = 0; c < 3; ++c) {
    r.ow[c] = omega * w[c];
    r.b[c] = 4.5 * omega * w[c];
    r.t[c] = 3.0 * omega_odd * w[c];
    r.gu[c] = 3.0 * (1.0 - 0.5 * omega) * w[c];
  }
  // n1 ow[1] and n2 ow[2] are multiples of the unit of ow[0], m t[2] one of that of 2 t[1]
  const double q0 = ulp(r.ow[0]), q1 = ulp(r.t[1]);
  r.ow[1] = multiple(r.ow[1], flat ? 0.25 * q0 : 0.5 * q0);
  r.ow[2] = multiple(r.ow[2], 0.25 * q0);
  r.t[2] = multiple(r.t[2], 2.0 * q1 / m);
  // 1 - keep - (n1 ow[1] + n2 ow[2]): both products are exact, the sum's rounding error
  // is taken along
  const double a = n1 * r.ow[1], b = n2 * r.ow[2], s = a + b, bb = s - a;
  const double e = (a - (s - bb)) + (b - bb);
  r.ow[0] = ((1.0 - r.keep) - s) - e;
  r.t[1] = 0.5 * ((1.0 - 2.0 * r.odd) - m * r.t[2]);
  return r;
}

}  // namespace olb
