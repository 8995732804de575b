// Learned interpolation weights per coarse cell (FP64, one rounding per
// operation): Dendy's edge sums split by the network's logits, and Dendy's
// centre formula (the local row solve) with those edge weights.  delta = 0
// gives Dendy's weights exactly.  Planes and weights may live in global or
// shared memory: the same functions serve bmg_setup's learned level 0, the
// test-vector loss and the per-crop two-grid training kernel.
#pragma once

#include "common.cuh"
#include "learned.h"

namespace bmg {
namespace learned {

// Logit k of interior coarse point (ic, jc); 0 for a ghost coarse point or
// without logits (delta = NULL: Dendy's weights).
__device__ __forceinline__ double delta_at(const float* delta, int nc, int ic, int jc, int k) {
  if (delta == nullptr || ic < 1 || jc < 1 || ic > nc || jc > nc) return 0.0;
  return (double)delta[((size_t)(jc - 1) * nc + (ic - 1)) * MLP_OUT + k];
}

// fl32(fl64(s / o)) for both feature sums s of a point over its diagonal o.  The
// quotients are formed to about 2^-39 from one reciprocal (the hardware's
// approximation and one Newton step) and rounded to 24 bits on the bit pattern;
// only where a quotient lies within about 2^-36 of a rounding boundary, or outside
// 2^[-100, 100], is it divided out: six FP64 operations a point, against about
// 22 with two divisions (FP64 is what bounds the features).
static __device__ __noinline__ float feature_slow(double s, double o) { return __double2float_rn(rdiv(s, o)); }

__device__ __forceinline__ float feature_round(double q, double s, double o) {
  const unsigned hi = (unsigned)__double2hiint(q), lo = (unsigned)__double2loint(q), e = (hi >> 20) & 0x7ffu;
  const unsigned low = lo & 0x1fffffffu;           // the 29 bits that rounding drops; half is 2^28
  if (e - 923u > 200u || low - 0x0ffe0000u <= 0x40000u) return feature_slow(s, o);
  const unsigned bits = (hi & 0x80000000u) | ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
  return __uint_as_float(bits + (low >> 28));      // (a carry moves into the exponent, as it should)
}

__device__ __forceinline__ float2 feature_pair(double w, double e, double s, double n, double o) {
  const double sx = radd(w, e), sy = radd(s, n);
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;\n" : "=d"(y) : "d"(o));
  y = __fma_rn(y, __fma_rn(-o, y, 1.0), y);
  return make_float2(feature_round(sx * y, sx, o), feature_round(sy * y, sy, o));
}

// Share of the first of an edge point's two coarse points, u_1 / (u_1 + u_2) with
// u_k = c_k exp(l_k): both terms divided by exp(l_1), one exponential (about 25
// FP64 operations) instead of two.  Logits 600 and more apart (or NaN) take the
// two exponentials: exp(l_2 - l_1) then leaves the FP64 range, or comes so near
// its ends that a product with c_2 may, and with a c_k of zero (no coupling to
// that side) the share would be NaN.  The test is on the bit pattern.
static __device__ __noinline__ double first_share_apart(double c1, double c2, double l1, double l2) {
  const double u1 = rmul(c1, exp(l1)), u2 = rmul(c2, exp(l2));
  return rdiv(u1, radd(u1, u2));
}

__device__ __forceinline__ double first_share(double c1, double c2, double l1, double l2) {
  const double d = rsub(l2, l1);
  if (((unsigned)__double2hiint(d) & 0x7fffffffu) >= 0x4082c000u) return first_share_apart(c1, c2, l1, l2);
  return rdiv(c1, radd(c1, rmul(c2, exp(d))));
}

// Edge points of cell (ic, jc), 0 <= ic, jc <= nc+1: x-edge (2ic-1, 2jc) between
// (ic-1, jc) [its E logit] and (ic, jc) [its W logit]; y-edge (2ic, 2jc-1)
// between (ic, jc-1) [N logit] and (ic, jc) [S logit].  An edge point keeps
// Dendy's total weight S_D = -(col_1 + col_2)/D and splits it in the shares
// u_k = -col_k exp(logit).  aux (optional, 4 coarse planes) keeps S_D and the
// first share q for the gradient.
__device__ __forceinline__ void edge_cell(const Planes<double>& A, int ld, int nc, const float* delta, int ic, int jc,
                                          double* ci, double* aux) {
  const int ldc = nc + 2;
  const size_t psc = plane_size(nc), pc = (size_t)jc * ldc + ic;
  double ll = 0, lr = 0, lb = 0, la = 0, sdx = 0, qx = 0, sdy = 0, qy = 0;
  if (ic >= 1 && jc >= 1 && jc <= nc) {
    size_t p = (size_t)(2 * jc) * ld + (2 * ic - 1);
    double colW = radd(radd(A.a<5>(p, ld), A.a<1>(p, ld)), A.a<7>(p, ld));
    double colE = radd(radd(A.a<8>(p, ld), A.a<2>(p, ld)), A.a<6>(p, ld));
    double D = radd(radd(A.a<3>(p, ld), A.a<0>(p, ld)), A.a<4>(p, ld));
    sdx = -rdiv(radd(colW, colE), D);
    qx = first_share(-colW, -colE, delta_at(delta, nc, ic - 1, jc, 1), delta_at(delta, nc, ic, jc, 0));
    ll = rmul(sdx, qx);
    lr = rmul(sdx, rsub(1.0, qx));
  }
  if (ic >= 1 && ic <= nc && jc >= 1) {
    size_t p = (size_t)(2 * jc - 1) * ld + 2 * ic;
    double rowS = radd(radd(A.a<5>(p, ld), A.a<3>(p, ld)), A.a<8>(p, ld));
    double rowN = radd(radd(A.a<7>(p, ld), A.a<4>(p, ld)), A.a<6>(p, ld));
    double D = radd(radd(A.a<1>(p, ld), A.a<0>(p, ld)), A.a<2>(p, ld));
    sdy = -rdiv(radd(rowS, rowN), D);
    qy = first_share(-rowS, -rowN, delta_at(delta, nc, ic, jc - 1, 3), delta_at(delta, nc, ic, jc, 2));
    lb = rmul(sdy, qy);
    la = rmul(sdy, rsub(1.0, qy));
  }
  ci[CI_LL * psc + pc] = ll;
  ci[CI_LR * psc + pc] = lr;
  ci[CI_LB * psc + pc] = lb;
  ci[CI_LA * psc + pc] = la;
  if (aux) {
    aux[0 * psc + pc] = sdx;
    aux[1 * psc + pc] = qx;
    aux[2 * psc + pc] = sdy;
    aux[3 * psc + pc] = qy;
  }
}

// Dendy's centre formula of cell (ic, jc) with the edge planes of ci (which
// must be complete for the neighbouring cells first).
__device__ __forceinline__ void centre_cell(const Planes<double>& A, int ld, int nc, int ic, int jc, double* ci) {
  const int ldc = nc + 2;
  const size_t psc = plane_size(nc), pc = (size_t)jc * ldc + ic;
  if (ic == 0 || jc == 0) {
    for (int k = 0; k < 4; ++k) ci[k * psc + pc] = 0.0;
    return;
  }
  size_t p = (size_t)(2 * jc - 1) * ld + (2 * ic - 1);
  double aO = A.a<0>(p, ld), aW = A.a<1>(p, ld), aE = A.a<2>(p, ld), aS = A.a<3>(p, ld), aN = A.a<4>(p, ld);
  double aSW = A.a<5>(p, ld), aNE = A.a<6>(p, ld), aNW = A.a<7>(p, ld), aSE = A.a<8>(p, ld);
  double lb_w = ci[CI_LB * psc + pc - 1], la_w = ci[CI_LA * psc + pc - 1];
  double lb_e = ci[CI_LB * psc + pc], la_e = ci[CI_LA * psc + pc];
  double ll_s = ci[CI_LL * psc + pc - ldc], lr_s = ci[CI_LR * psc + pc - ldc];
  double ll_n = ci[CI_LL * psc + pc], lr_n = ci[CI_LR * psc + pc];
  // one division and four quotients by the same divisor (quot rounds as the division does)
  double yl;
  const double y = quot_recip(aO, &yl);
  ci[CI_LSW * psc + pc] = -quot(radd(radd(aSW, rmul(aW, lb_w)), rmul(aS, ll_s)), aO, y, yl);
  ci[CI_LSE * psc + pc] = -quot(radd(radd(aSE, rmul(aE, lb_e)), rmul(aS, lr_s)), aO, y, yl);
  ci[CI_LNW * psc + pc] = -quot(radd(radd(aNW, rmul(aW, la_w)), rmul(aN, ll_n)), aO, y, yl);
  ci[CI_LNE * psc + pc] = -quot(radd(radd(aNE, rmul(aE, la_e)), rmul(aN, lr_n)), aO, y, yl);
}

}  // namespace learned
}  // namespace bmg
