// Closures of the free-slip top (open channel, top_bc = 1; paper Sec. 3.1).
// The tau rows n >= 2 are those of the no-slip channel, so elimination leaves
// each parity affine in its lowest coefficient, f = P + x Q (P_0 = 0, Q_0 = 1);
// only the wall rows change, and they couple the two parities:
//   omega_y, W:  f(-1) = S_e - S_o,  Df(+1) = S2_e + S2_o
//                (S = sum over the parity of f_n, S2 = sum of n^2 f_n);
//   U:           the same two rows and the flow rate, with the response to
//                the unknown forcing (even parity);
//   v:           v(+-1) stay Dirichlet per parity; phi = P + c vh per parity,
//                and D^2 v(+1) = A_e + A_o, Dv(-1) = -B_e + B_o
//                (A = sum n^2 (n^2 - 1) / 3 v_n, B = sum n^2 v_n) fix c_e, c_o.
// With the shifted unknowns f' = f + cc f_old every row's value is cc times
// that row applied to the old field.  The threads of both parities solve the
// same closure, summing in parity order, so both find the same coefficients.
#pragma once

#include "common.cuh"

namespace chdns {

// a11 x1 + a12 x2 = b1, a21 x1 + a22 x2 = b2 (Cramer's rule)
__device__ __forceinline__ void solve2(double a11, double a12, double a21, double a22, double b1, double b2,
                                       double* x1, double* x2) {
  const double id = 1.0 / fma_rn(a11, a22, -mul_rn(a12, a21));
  *x1 = mul_rn(fma_rn(b1, a22, -mul_rn(a12, b2)), id);
  *x2 = mul_rn(fma_rn(a11, b2, -mul_rn(a21, b1)), id);
}

// Dirichlet bottom and Neumann top rows over the two parities of omega_y or W.
// se, so: {sum P, sum n^2 P, sum f_old, sum n^2 f_old} of the even and odd
// parity; q*: the table sums sum Q and sum n^2 Q.
__device__ __forceinline__ void close_neumann_top(const double* se, const double* so, double qe, double qo,
                                                  double q2e, double q2o, double cc, double* xe, double* xo) {
  solve2(qe, -qo, q2e, q2o, fma_rn(cc, se[2] - so[2], -(se[0] - so[0])), fma_rn(cc, se[3] + so[3], -(se[1] + so[1])),
         xe, xo);
}

// Influence coefficients of v: se, so = {A_p, B_p, A_old, B_old}; a*, b*: A
// and B of the homogeneous solutions vh of the two parities.
__device__ __forceinline__ void close_free_slip_v(const double* se, const double* so, double ae, double ao,
                                                  double be, double bo, double cc, double* ce, double* co) {
  solve2(ae, ao, -be, bo, fma_rn(cc, se[2] + so[2], -(se[0] + so[0])), fma_rn(cc, so[3] - se[3], -(so[1] - se[1])),
         ce, co);
}

// Mean U at constant flow rate: unknowns (x_e, x_o, forcing).  se = {sum P,
// sum n^2 P, sum U_old, sum n^2 U_old, int P, int U_old}, so = the first four
// of the odd parity; q*: sum Q, sum n^2 Q; wq: int Q_e; u*: sum, sum n^2 and
// int of the forcing response (even).  int = sum of 2 / (1 - n^2) x_n.
__device__ __forceinline__ void close_free_slip_mean(const double* se, const double* so, double qe, double qo,
                                                     double q2e, double q2o, double wq, double us, double u2,
                                                     double uw, double cc, double flux, double* xe, double* xo,
                                                     double* fc) {
  const double a11 = qe, a12 = -qo, a13 = us;
  const double a21 = q2e, a22 = q2o, a23 = u2;
  const double a31 = wq, a32 = 0.0, a33 = uw;
  const double b1 = fma_rn(cc, se[2] - so[2], -(se[0] - so[0]));
  const double b2 = fma_rn(cc, se[3] + so[3], -(se[1] + so[1]));
  const double b3 = fma_rn(cc, se[5], flux) - se[4];
  // 2 x 2 minors (x y - z w, fused on the first product)
  auto det2 = [](double x, double y, double z, double w) { return fma_rn(x, y, -mul_rn(z, w)); };
  const double m1 = det2(a22, a33, a23, a32), m2 = det2(a21, a33, a23, a31), m3 = det2(a21, a32, a22, a31);
  const double id = 1.0 / fma_rn(a13, m3, fma_rn(a11, m1, -mul_rn(a12, m2)));
  *xe = mul_rn(fma_rn(a13, det2(b2, a32, a22, b3), fma_rn(b1, m1, -mul_rn(a12, det2(b2, a33, a23, b3)))), id);
  *xo = mul_rn(fma_rn(a13, det2(a21, b3, b2, a31), fma_rn(a11, det2(b2, a33, a23, b3), -mul_rn(b1, m2))), id);
  *fc = mul_rn(fma_rn(b1, m3, fma_rn(a11, det2(a22, b3, b2, a32), -mul_rn(a12, det2(a21, b3, b2, a31)))), id);
}

}  // namespace chdns
