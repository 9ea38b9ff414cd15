// Derivative of a Slater-Koster sp block with respect to the bond vector, contracted with the block's rho and pi
// (device code shared by the force kernels).
#pragma once

#include <math.h>

namespace mka {

// out = -2 sum_{c,r} (rho[c][r] dH[c][r]/dd - pi[c][r] dS[c][r]/dd) for the two-centre block of displacement d (s, px,
// py, pz order; rho and pi: 16 entries at 4 c + r):
//   [s][s] = ss s(r), [s][p_k] = c_k sp s(r), [p_k][s] = -[s][p_k],
//   [p_k][p_m] = c_k c_m (pps - ppp) s(r) + delta_km ppp s(r), s(r) = exp(-2 (r/d0 - 1)), c = d / r.
// The sums over the entries are taken first: with X_v = rho Vh_v - pi Vs_v, a = X_ss[s][s], b_k = X_sp[s][p_k] -
// X_sp[p_k][s], M = X_pps - X_ppp and q = (M + M^T) c, the derivative with respect to d_l is
//   s'(r) c_l (a + b.c + c.Mc + tr X_ppp) + s(r) / r (b_l + q_l - c_l (b.c + 2 c.Mc)).
// One thread a block and one square root, exponential and division: the derivative of each entry by itself took 32 of
// each and five times the FP64 operations.
__device__ __forceinline__ void sk_block_force(const double d[3], const double* Vh, const double* Vs, double d0,
                                               const double* rho, const double* pi, double out[3]) {
  const double r = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
  const double ir = 1.0 / r;
  const double c[3] = {d[0] * ir, d[1] * ir, d[2] * ir};
  const double s = exp(-2.0 * (r / d0 - 1.0));
  const double sr = -(2.0 / d0) * s;      // ds/dr
  const double sir = s * ir;
  const double dh = Vh[2] - Vh[3], ds = Vs[2] - Vs[3];
  double q[3] = {0.0, 0.0, 0.0}, b[3];
  double trh = 0.0, trs = 0.0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    b[k] = Vh[1] * (rho[k + 1] - rho[4 * (k + 1)]) - Vs[1] * (pi[k + 1] - pi[4 * (k + 1)]);
    trh += rho[5 * (k + 1)];
    trs += pi[5 * (k + 1)];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const double x = dh * rho[4 * (k + 1) + m + 1] - ds * pi[4 * (k + 1) + m + 1];
      q[k] += x * c[m];
      q[m] += x * c[k];
    }
  }
  const double bc = b[0] * c[0] + b[1] * c[1] + b[2] * c[2];
  const double cm2 = q[0] * c[0] + q[1] * c[1] + q[2] * c[2];   // 2 c.Mc
  const double a = Vh[0] * rho[0] - Vs[0] * pi[0] + (Vh[3] * trh - Vs[3] * trs);
  const double along = sr * (a + bc + 0.5 * cm2) - sir * (bc + cm2);
#pragma unroll
  for (int l = 0; l < 3; ++l) out[l] = -2.0 * (along * c[l] + sir * (b[l] + q[l]));
}

}  // namespace mka
