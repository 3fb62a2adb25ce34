// The tridiagonal solve behind chi(omega) (Eqs. resolvent_Liouvillian_Lanczos_q and
// post_processing), shared by tdlz_spectrum and tdlz_spectrum_noalloc.
//
// Bound by the FP64 issue rate of one warp: each of an SM's four schedulers starts one FP64
// warp instruction per 64 clocks, whatever the number of active lanes (the four together
// one per 19), so a solve takes 64 clocks x the instructions of a step x the steps until
// the 608 schedulers are full.  Hence one thread per (chain, omega, left vector) with the
// continuant recomputed by each (16 instructions a step instead of 28 for all three left
// vectors: 282 warps for 3 chains x 1001 frequencies), in blocks of one warp so that they
// spread over the SMs.
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

// 2^-e of the upper word `mag` of the largest component; 1 for zero and non-finite values
__device__ __forceinline__ double spec_pow2(int mag) {
  const int e = (mag >> 20) - 1023;
  return e > -1000 && e < 1000 ? __hiloint2double((1023 - e) << 20, 0) : 1.0;
}

// sum_i conj(z_i) x_i for (zw - T) x = e_1 with the m x m tridiagonal T (diagonal alpha,
// sub-diagonal beta, super-diagonal gamma) and `tail` subtracted from the last diagonal
// entry (the continued fraction of an extrapolated part; zero without one).
//
// With D_i the determinant of rows and columns i..m,
//   D_i = (zw - alpha_i) D_{i+1} - beta_i gamma_i D_{i+2},
//   x_i = beta_1 .. beta_{i-1} D_{i+1} / D_1,
// so the sum is A_1 / D_1 with A_i = conj(z_i) D_{i+1} + beta_i A_{i+1}: one sweep from the
// last row up, no division, no pivots and no stored rows.  The D computed this way are the
// exact ones of a matrix whose entries differ by rounding errors (each step's errors can be
// put on its own alpha and beta gamma), so the solve is at least as stable as elimination
// with partial pivoting; measured against extended precision at 1500 steps: 3.6e-16
// (non-Hermitian chains) and 1.5e-16 (alternating signs) of the norm, pivoted elimination
// 6.6e-16 and 1.9e-16.  D and A share one power-of-two scale, which the ratio drops.
// Whole calls, 3 chains x 1500 steps x 1001 frequencies: 9.31 ms with pivoted elimination
// over stored rows, 2.80 ms without the rows, 1.27 ms in this form.
__device__ __forceinline__ double2 tridiag_chi(int m, const double2 *__restrict__ al,
                                               const double *__restrict__ be,
                                               const double2 *__restrict__ ga,
                                               const double2 *__restrict__ z, double2 zw,
                                               double2 tail) {
  double2 d1 = make_double2(zw.x - al[m - 1].x - tail.x, zw.y - al[m - 1].y - tail.y);  // D_m
  double2 d2 = make_double2(1.0, 0.0);
  double2 A = make_double2(z[m - 1].x, -z[m - 1].y);
  // coefficients of the next row, loaded one step ahead
  const int i0 = m > 1 ? m - 2 : 0;
  double2 an = al[i0], gn = ga[i0], zn = z[i0];
  double bn = be[i0];
  for (int i = m - 2; i >= 0; --i) {
    const double2 d = make_double2(zw.x - an.x, zw.y - an.y), zv = zn;
    const double2 bc = make_double2(bn * gn.x, bn * gn.y);
    const double b = bn;
    const int in = i > 0 ? i - 1 : 0;
    an = al[in];
    gn = ga[in];
    zn = z[in];
    bn = be[in];
    // conj(z) D + beta A
    A = make_double2(fma(zv.x, d1.x, fma(zv.y, d1.y, b * A.x)),
                     fma(zv.x, d1.y, fma(-zv.y, d1.x, b * A.y)));
    const double2 t = spec_mul(d, d1);
    const double2 d0 = spec_nfma(t, bc, d2);
    d2 = d1;
    d1 = d0;
    const int mag = max(spec_mag(d1), spec_mag(d2));
    if (mag < (823 << 20) || mag > (1223 << 20)) {  // beyond 2^+-200 (seldom)
      const double sc = spec_pow2(mag);
      d1 = make_double2(d1.x * sc, d1.y * sc);
      d2 = make_double2(d2.x * sc, d2.y * sc);
      A = make_double2(A.x * sc, A.y * sc);
    }
  }
  return spec_cdiv(A, d1);
}

}  // namespace tdlz
