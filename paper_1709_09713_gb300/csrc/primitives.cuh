// primitives.cuh -- velocities, pressure and temperature of a point (Eqs. 4-5) in
// binary64, for the comparison classes, which keep them in arrays.
#pragma once

#include "fpconv.cuh"

namespace sbli {

__device__ __forceinline__ bool is_finite_f64(double x) { return (~__double2hiint(x) & 0x7FF00000) != 0; }

// u_i = m_i / rho, p' and T' (Eqs. 4-5) in deviation form, for the kernels that keep
// them in arrays: one reciprocal for the four quotients instead of four divisions,
// which take over, in a function of their own, where a quotient is not finite (an infinite
// density divides to 0).  128^3 store-all stage 1.049 ms without that and 1.050 with it;
// a check and an inlined division at each quotient 1.164.
struct Primitives {
  double u[3], p, t;
};
template <typename Q>
__device__ __forceinline__ Primitives primitives_of(double rho_p, double m0, double m1, double m2, double E, double gm1,
                                                    double gM2, const Q& quotient) {
  Primitives r;
  r.u[0] = quotient(m0);
  r.u[1] = quotient(m1);
  r.u[2] = quotient(m2);
  r.p = gm1 * (E - 0.5 * (1.0 + rho_p) * (r.u[0] * r.u[0] + r.u[1] * r.u[1] + r.u[2] * r.u[2]));
  r.t = quotient(gM2 * r.p - rho_p);
  return r;
}
static __device__ __noinline__ Primitives primitives_by_division(double rho_p, double m0, double m1, double m2, double E,
                                                                 double gm1, double gM2) {
  return primitives_of(rho_p, m0, m1, m2, E, gm1, gM2, [&](double x) { return x / (1.0 + rho_p); });
}
__device__ __forceinline__ Primitives primitives_f64(double rho_p, double m0, double m1, double m2, double E, double gm1,
                                                     double gM2) {
  const double rho = 1.0 + rho_p, rinv = rcp_newton_f64(rho);
  Primitives r =
      primitives_of(rho_p, m0, m1, m2, E, gm1, gM2, [&](double x) { return corrected_quotient(x, rho, rinv); });
  if (!(is_finite_f64(r.u[0]) && is_finite_f64(r.u[1]) && is_finite_f64(r.u[2]) && is_finite_f64(r.t)))
    r = primitives_by_division(rho_p, m0, m1, m2, E, gm1, gM2);
  return r;
}

}  // namespace sbli
