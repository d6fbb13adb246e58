// The branch subproblem of the linear feasibility projection (linfeas.cu): a
// convex QP in v = (w_i, w_j | wR, wI) with Hessian
//
//   rho F'F + diag(rho, rho | 2, 2),   F the four flow rows over v,
//
// and bounds on w_i, w_j.  Host and device code: the kernels call it per
// branch, and the same code compiles on the host for the CPU tests.
//
// wR and wI have no bounds and their block is a multiple d I of the identity
// (the two columns of F are orthogonal and of equal norm), so they are
// eliminated: with T_i, T_j the off-diagonal blocks over d, w = (w_i, w_j)
// minimises 1/2 w'Sw + s'w over its box with S the Schur complement.
//
// S is nearly singular along (1, 1) for a short line: its eigenvalues are about
// rho and rho |Y|^2, so rounding of s moves w along that direction by about
// |Y|^2 2^-53, which changes the flows F v by |Y|^2 2^-53 only -- as long as w_i
// and w_j move together.  Three things keep it so:
//   - S and its determinant are formed without cancellation (lf_constants);
//   - the unconstrained minimiser comes from the LDL' factors, w_i from w_j,
//     and not from the inverse, whose two rows round independently;
//   - the active bounds are decided by the signs of the gradient, not by
//     comparing objective values, which agree to rounding near a corner, and
//     whatever a sign decides wrongly within rounding, the variable left free
//     is the minimiser for the value of the other.
// Against 128-bit arithmetic, 100,000 minimisers within 1e-1 to 1e-14 of a
// bound, |Y| 30 / 300 / 3,000: largest error of v 7e-14 / 1e-11 / 9e-10 and of
// the flows 4e-14 / 3e-12 / 2e-10.
#pragma once

#include "line_qp.cuh"

namespace acopf {

// Constants of a branch: T (0-3), l = S12/S11, 1/S11, S11/det S (4-6), 1/d (7),
// 2 wR0, 2 wI0 (8, 9), bounds of w_i and w_j (10-13)
constexpr int kLfBranch = 14;

// The first eight from the admittances Y = (gii bii gij bij gji bji gjj bjj).
// |T_i d|^2 = rho^2 |Yii|^2 |Yij|^2, which turns S11 = rho (|Yii|^2 + 1) - d
// |T_i|^2 and the determinant into sums of positive terms:
//   S11 = rho (1 + e_i), e_i = |Yii|^2 (rho |Yji|^2 + 2) / d, and e_j likewise;
//   det S = rho^2 (1 + e_i + e_j + 2 |Yii|^2 |Yjj|^2 / d) + d^2 (T_i x T_j)^2.
ACOPF_HD inline void lf_constants(const double Y[8], double rho, double c[8]) {
  const double gii = Y[0], bii = Y[1], gij = Y[2], bij = Y[3], gji = Y[4], bji = Y[5], gjj = Y[6], bjj = Y[7];
  const double nii = gii * gii + bii * bii, njj = gjj * gjj + bjj * bjj;
  const double nij = gij * gij + bij * bij, nji = gji * gji + bji * bji;
  const double d = rho * (nij + nji) + 2.0, r = rho / d;
  c[0] = r * (gii * gij + bii * bij);
  c[1] = r * (gii * bij - bii * gij);
  c[2] = r * (gjj * gji + bjj * bji);
  c[3] = r * (bjj * gji - gjj * bji);
  const double ei = nii * (rho * nji + 2.0) / d, ej = njj * (rho * nij + 2.0) / d;
  const double x = d * (c[0] * c[3] - c[1] * c[2]);
  const double s11 = rho * (1.0 + ei), s12 = -d * (c[0] * c[2] + c[1] * c[3]);
  const double det = rho * rho * (1.0 + ei + ej + 2.0 * nii * (njj / d)) + x * x;
  c[4] = s12 / s11;
  c[5] = 1.0 / s11;
  c[6] = s11 / det;
  c[7] = 1.0 / d;
}

// w when the unconstrained minimiser (given in wi, wj) lies outside the box.
// l, i1, i2: constants 4 to 6; S22 = det / S11 + S12^2 / S11.  The function of
// w_i that is left when w_j is minimised out is convex: its slope at the two
// bounds tells whether w_i lies on one; otherwise w_j does.
ACOPF_HD inline void lf_edges(double l, double i1, double i2, double si, double sj, double li, double hi, double lj,
                              double hj, double& wi, double& wj) {
  const double s11 = 1.0 / i1, s12 = l * s11, i22 = 1.0 / (1.0 / i2 + l * s12);
  double v = clampv(-(sj + s12 * li) * i22, lj, hj);
  if (s11 * li + s12 * v + si >= 0.0) {
    wi = li;
    wj = v;
    return;
  }
  v = clampv(-(sj + s12 * hi) * i22, lj, hj);
  if (s11 * hi + s12 * v + si <= 0.0) {
    wi = hi;
    wj = v;
    return;
  }
  const double s22 = 1.0 / i2 + l * s12;
  const double ul = -(si * i1 + l * lj), uh = -(si * i1 + l * hj);
  if (s12 * ul + s22 * lj + sj >= 0.0) {
    wi = ul;
    wj = lj;
    if (ul >= li && ul <= hi) return;
  } else if (s12 * uh + s22 * hj + sj <= 0.0) {
    wi = uh;
    wj = hj;
    if (uh >= li && uh <= hi) return;
  }
  // the signs disagree within rounding: each variable in turn for the other's value
  wi = clampv(wi, li, hi);
  wj = clampv(-(sj + s12 * wi) * i22, lj, hj);
  wi = clampv(-(si * i1 + l * wj), li, hi);
}

// v from y = lambda - rho z of the two ends' flows and voltage copies: (w_i,
// w_j, wR, wI); edges is lf_edges (a parameter, so that the kernel can call it
// out of line)
template <typename Edges>
ACOPF_HD inline void lf_branch(const double Y[8], const double c[kLfBranch], const double yi[3], const double yj[3],
                               double v[4], const Edges& edges) {
  const double gii = Y[0], bii = Y[1], gij = Y[2], bij = Y[3], gji = Y[4], bji = Y[5], gjj = Y[6], bjj = Y[7];
  // gradient at v = 0: F' y_f + (copies, -2 wR0, -2 wI0)
  const double ci = yi[2] + gii * yi[0] - bii * yi[1];
  const double cj = yj[2] + gjj * yj[0] - bjj * yj[1];
  const double cr = gij * yi[0] - bij * yi[1] + gji * yj[0] - bji * yj[1] - c[8];
  const double cm = bij * yi[0] + gij * yi[1] - bji * yj[0] - gji * yj[1] - c[9];
  const double si = ci - c[0] * cr - c[1] * cm;
  const double sj = cj - c[2] * cr - c[3] * cm;
  double wj = -c[6] * (sj - c[4] * si);
  double wi = -(si * c[5] + c[4] * wj);
  if (!(wi >= c[10] && wi <= c[11] && wj >= c[12] && wj <= c[13]))
    edges(c[4], c[5], c[6], si, sj, c[10], c[11], c[12], c[13], wi, wj);
  v[0] = wi;
  v[1] = wj;
  v[2] = -(c[7] * cr + c[0] * wi + c[2] * wj);
  v[3] = -(c[7] * cm + c[1] * wi + c[3] * wj);
}

}  // namespace acopf
