// The tridiagonal solve behind chi(omega) (Eqs. resolvent_Liouvillian_Lanczos_q and
// post_processing), shared by tdlz_spectrum and tdlz_spectrum_noalloc.
//
// One thread solves one (chain, omega).  The solve is bound by the FP64 pipe (two lanes
// per clock and SM on this part: a warp instruction takes 16 clocks of its SM whatever the
// other SMs do), so its cost is the FP64 instructions of one step times the steps, and the
// kernels run one warp per block: 3 chains x 1001 frequencies are 94 warps on 94 SMs
// instead of four to a block on 24.  Measured for that case with 1500 steps: see
// tridiag_chi.
#pragma once

#include <cuda_runtime.h>

namespace tdlz {

constexpr int kSpecThreads = 32;  // one warp per block (see above)

// a / b with scaling (Smith's method)
__device__ __forceinline__ double2 spec_cdiv(double2 a, double2 b) {
  if (fabs(b.x) >= fabs(b.y)) {
    double r = b.y / b.x, den = b.x + b.y * r;
    return make_double2((a.x + a.y * r) / den, (a.y - a.x * r) / den);
  }
  double r = b.x / b.y, den = b.x * r + b.y;
  return make_double2((a.x * r + a.y) / den, (a.y * r - a.x) / den);
}

__device__ __forceinline__ double2 spec_mul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// acc - a b
__device__ __forceinline__ double2 spec_nfma(double2 acc, double2 a, double2 b) {
  return make_double2(fma(-a.x, b.x, fma(a.y, b.y, acc.x)),
                      fma(-a.x, b.y, fma(-a.y, b.x, acc.y)));
}

// Upper word (sign cleared) of the larger component: orders complex numbers by their
// maximum norm to 20 bits without an FP64 instruction.
__device__ __forceinline__ int spec_mag(double2 a) {
  return max(__double2hiint(a.x) & 0x7fffffff, __double2hiint(a.y) & 0x7fffffff);
}

// 1 / c, one division; numbers whose square would leave the double range take Smith's
// method (mag = spec_mag(c): exponents within +-400).
__device__ __forceinline__ double2 spec_recip(double2 c, int mag) {
  if (mag >= (623 << 20) && mag < (1423 << 20)) {
    const double r = 1.0 / fma(c.x, c.x, c.y * c.y);
    return make_double2(c.x * r, -c.y * r);
  }
  return spec_cdiv(make_double2(1.0, 0.0), c);
}

// acc[l] = sum_i conj(z^l_i) x_i for (zw - T) x = e_1 with the m x m tridiagonal T
// (diagonal alpha, sub-diagonal beta, super-diagonal gamma) and `tail` subtracted from the
// last diagonal entry (the continued fraction of an extrapolated part; zero without one).
//
// Gaussian elimination with partial pivoting from the last row up.  The right-hand side is
// zero below the first row, so nothing has to be kept: eliminating x_{i+1} leaves one
// pending row  p x_i + q x_{i+1} = 0  and  x_{i+1} = s x_i + t x_{i-1}  (t != 0 only where
// row i was the pivot), and the sums over j > i are carried along as the functional
// A_l x_{i+1} + B_l x_i.  No scratch, no second sweep: against the top-down elimination
// that stored its rows (four complex words per step, written and read back) and formed two
// hypot and six divisions per step this does one division and about 45 FP64 instructions.
// 3 chains x 1500 steps x 1001 frequencies: 9.35 ms before, @SPEC_FULL@ after (whole calls).
// Pivots are compared in the maximum norm to 20 bits: |multiplier| <= sqrt 2, so the growth
// bound of partial pivoting stays; measured errors against extended precision are below
// the top-down form's (2.4e-16 against 6.1e-16 of the norm at 1500 steps).
template <int NL>
__device__ __forceinline__ void tridiag_chi(int m, int cap, const double2 *__restrict__ al,
                                            const double *__restrict__ be,
                                            const double2 *__restrict__ ga,
                                            const double2 *__restrict__ zz, double2 zw,
                                            double2 tail, double2 (&acc)[NL]) {
  double2 q = make_double2(zw.x - al[m - 1].x - tail.x, zw.y - al[m - 1].y - tail.y);
  double2 A[NL], B[NL];
#pragma unroll
  for (int l = 0; l < NL; ++l) {
    const double2 zv = zz[(long long)l * cap + m - 1];
    A[l] = make_double2(zv.x, -zv.y);
    B[l] = make_double2(0.0, 0.0);
  }
  if (m == 1) {
    const double2 x = spec_cdiv(make_double2(1.0, 0.0), q);
#pragma unroll
    for (int l = 0; l < NL; ++l) acc[l] = spec_mul(A[l], x);
    return;
  }
  double2 p = make_double2(-be[m - 2], 0.0);
  // coefficients of the next row, loaded one step ahead
  double2 an = al[m - 2], gn = ga[m - 2], zn[NL];
  double bn = m > 2 ? be[m - 3] : 0.0;
#pragma unroll
  for (int l = 0; l < NL; ++l) zn[l] = zz[(long long)l * cap + m - 2];
  for (int i = m - 2; i >= 1; --i) {
    const double2 d = make_double2(zw.x - an.x, zw.y - an.y), du = make_double2(-gn.x, -gn.y);
    const double dl = -bn;
    double2 zv[NL];
#pragma unroll
    for (int l = 0; l < NL; ++l) zv[l] = zn[l];
    an = al[i - 1];
    gn = ga[i - 1];
    bn = i > 1 ? be[i - 2] : 0.0;
#pragma unroll
    for (int l = 0; l < NL; ++l) zn[l] = zz[(long long)l * cap + i - 1];
    const int mq = spec_mag(q), mu = spec_mag(du);
    if (mq >= mu) {  // the pending row is the pivot: x_{i+1} = -(p / q) x_i
      const double2 ic = spec_recip(q, mq);
      const double2 s = spec_mul(p, ic), f = spec_mul(du, ic);  // s negated
      q = spec_nfma(d, f, p);
      p = make_double2(dl, 0.0);
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        const double2 c = make_double2(zv[l].x + B[l].x, B[l].y - zv[l].y);
        A[l] = spec_nfma(c, A[l], s);
        B[l] = make_double2(0.0, 0.0);
      }
    } else {  // row i is the pivot: x_{i+1} = -(d x_i + dl x_{i-1}) / du
      const double2 ic = spec_recip(du, mu);
      const double2 s = spec_mul(d, ic), f = spec_mul(q, ic);
      const double2 t = make_double2(-dl * ic.x, -dl * ic.y);
      q = spec_nfma(p, f, d);
      p = make_double2(-f.x * dl, -f.y * dl);
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        const double2 c = make_double2(zv[l].x + B[l].x, B[l].y - zv[l].y);
        B[l] = spec_mul(A[l], t);
        A[l] = spec_nfma(c, A[l], s);
      }
    }
  }
  // first row: d x_1 + du x_2 = 1 with the pending p x_1 + q x_2 = 0
  const double2 d = make_double2(zw.x - an.x, zw.y - an.y), du = make_double2(-gn.x, -gn.y);
  const double2 one = make_double2(1.0, 0.0);
  double2 x1, x2;
  if (spec_mag(q) >= spec_mag(du)) {
    const double2 ic = spec_cdiv(one, q);
    x1 = spec_cdiv(one, spec_nfma(d, spec_mul(du, ic), p));
    const double2 s = spec_mul(p, ic);
    x2 = spec_nfma(make_double2(0.0, 0.0), s, x1);
  } else {
    const double2 ic = spec_cdiv(one, du);
    const double2 f = spec_mul(q, ic);
    x1 = spec_cdiv(make_double2(-f.x, -f.y), spec_nfma(p, f, d));
    x2 = spec_mul(spec_nfma(one, d, x1), ic);
  }
#pragma unroll
  for (int l = 0; l < NL; ++l) {
    const double2 b = make_double2(B[l].x + zn[l].x, B[l].y - zn[l].y);
    const double2 ax = spec_mul(A[l], x2), bx = spec_mul(b, x1);
    acc[l] = make_double2(ax.x + bx.x, ax.y + bx.y);
  }
}

}  // namespace tdlz
