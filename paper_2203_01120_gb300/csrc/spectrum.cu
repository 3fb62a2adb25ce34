// chi(omega) from the Lanczos tridiagonal matrix (Eqs.
// resolvent_Liouvillian_Lanczos_q and post_processing), FP64 on the GPU.
//
// One thread per (chain, omega, left vector l) solves (omega + i eta - T) x = e_1 and
// forms chi_l = w n0 sum_i conj(z^l_i) x_i in the same sweep (spectrum_solve.cuh).
#include <cmath>

#include "spectrum.cuh"
#include "spectrum_solve.cuh"

namespace tdlz {

// 2 x 2 complex matrices as (x0 x1; x2 x3), scaled by a power of two so that repeated
// products stay in range (a Moebius map does not depend on the scale).
struct Mob {
  double2 x[4];
};

__device__ __forceinline__ Mob mob_mul(const Mob &a, const Mob &b) {
  const double2 zero = make_double2(0.0, 0.0);
  Mob r;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const double2 na = make_double2(-a.x[2 * i].x, -a.x[2 * i].y);
      const double2 nb = make_double2(-a.x[2 * i + 1].x, -a.x[2 * i + 1].y);
      r.x[2 * i + j] = spec_nfma(spec_nfma(zero, na, b.x[j]), nb, b.x[2 + j]);
    }
  int mag = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) mag = max(mag, spec_mag(r.x[i]));
  const double sc = spec_pow2(mag);
#pragma unroll
  for (int i = 0; i < 4; ++i) r.x[i] = make_double2(r.x[i].x * sc, r.x[i].y * sc);
  return r;
}

// v <- a v for the homogeneous coordinates v = (numerator, denominator)
__device__ __forceinline__ void mob_apply(const Mob &a, double2 (&v)[2]) {
  double2 n0 = spec_mul(a.x[0], v[0]), n1 = spec_mul(a.x[1], v[1]);
  double2 d0 = spec_mul(a.x[2], v[0]), d1 = spec_mul(a.x[3], v[1]);
  v[0] = make_double2(n0.x + n1.x, n0.y + n1.y);
  v[1] = make_double2(d0.x + d1.x, d0.y + d1.y);
  const double sc = spec_pow2(max(spec_mag(v[0]), spec_mag(v[1])));
#pragma unroll
  for (int i = 0; i < 2; ++i) v[i] = make_double2(v[i].x * sc, v[i].y * sc);
}

__global__ void __launch_bounds__(kSpecThreads) spectrum_kernel(SpecArgs a) {
  long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (tid >= (long long)a.nchain * a.nomega * a.nl) return;
  const long long ciw = tid / a.nl;
  const int l = (int)(tid - ciw * a.nl);
  const int c = (int)(ciw / a.nomega);
  const int iw = (int)(ciw - (long long)c * a.nomega);
  int m = a.steps[c];
  if (a.itermax0 > 0 && a.itermax0 < m) m = a.itermax0;
  double2 *out = a.chi + ((long long)c * a.nl + l) * a.nomega + iw;
  if (m <= 0) {
    *out = make_double2(0, 0);
    return;
  }
  const double2 *al = a.alpha + (long long)c * a.cap;
  const double *be = a.beta + (long long)c * a.cap;
  const double2 *ga = a.gamma + (long long)c * a.cap;
  const double2 *zz = a.z + ((long long)c * a.nl + l) * a.cap;
  double om = a.start + a.step * iw;
  double2 zw = make_double2(om, a.eta);
  // Extrapolated tail (Sec. 3.3): coefficients m..itermax-1 are the means of the
  // computed ones over [m/2, m) (per parity for the bi-constant form), z = 0
  // there; the tail enters through the backward continued fraction g and one
  // modified diagonal entry d_{m-1} -= beta_{m-1} gamma_{m-1} g.
  double2 tail = make_double2(0, 0);
  if (a.extrap != 0 && a.itermax > m && m >= 2) {
    double2 ca[2] = {{0, 0}, {0, 0}}, cg[2] = {{0, 0}, {0, 0}};
    double cb[2] = {0, 0};
    int cnt[2] = {0, 0};
    for (int j = m / 2; j < m; ++j) {
      int p = a.extrap == 2 ? (j & 1) : 0;
      ca[p].x += al[j].x;
      ca[p].y += al[j].y;
      cb[p] += be[j];
      cg[p].x += ga[j].x;
      cg[p].y += ga[j].y;
      cnt[p]++;
    }
    if (a.extrap != 2) {
      ca[1] = ca[0];
      cb[1] = cb[0];
      cg[1] = cg[0];
      cnt[1] = cnt[0];
    }
    Mob step[2];  // g_j = 1 / (zw - alpha_j - beta_j gamma_j g_{j+1}), j even and odd
    for (int p = 0; p < 2; ++p) {
      double inv = cnt[p] > 0 ? 1.0 / cnt[p] : 0.0;
      ca[p] = make_double2(ca[p].x * inv, ca[p].y * inv);
      cb[p] *= inv;
      cg[p] = make_double2(cg[p].x * inv, cg[p].y * inv);
      step[p].x[0] = make_double2(0, 0);
      step[p].x[1] = make_double2(1, 0);
      step[p].x[2] = make_double2(-cb[p] * cg[p].x, -cb[p] * cg[p].y);
      step[p].x[3] = make_double2(zw.x - ca[p].x, zw.y - ca[p].y);
    }
    // The tail's coefficients repeat with period two, so its itermax - m steps are a power
    // of one pair of steps, applied by binary powers (12 squarings for 5620 steps) instead
    // of one complex division each; relative error 9e-16 against 1.5e-15 of the serial
    // fraction at 380 + 5620 steps (both against extended precision).
    const int n = a.itermax - m;
    double2 v[2] = {{0, 0}, {1, 0}};  // g beyond the last step is 0
    if (n & 1) mob_apply(step[(a.itermax - 1) & 1], v);
    Mob pw = mob_mul(step[m & 1], step[(m + 1) & 1]);
    for (int h = n >> 1; h > 0; h >>= 1) {
      if (h & 1) mob_apply(pw, v);
      if (h > 1) pw = mob_mul(pw, pw);
    }
    const double2 g = spec_cdiv(v[0], v[1]);
    double2 bg = make_double2(be[m - 1] * ga[m - 1].x, be[m - 1] * ga[m - 1].y);
    tail = make_double2(bg.x * g.x - bg.y * g.y, bg.x * g.y + bg.y * g.x);
  }
  const double2 acc = tridiag_chi(m, al, be, ga, zz, zw, tail);
  double s = a.wk[c] * a.n0[c];
  *out = make_double2(s * acc.x, s * acc.y);
}

// S(w) = -Im sum_ab P_ab chi_ba(w), chi[a][b][w] = chi_ba (chain a, row b)  (Eq. S_def)
__global__ void structure_factor_kernel(const double2 *__restrict__ chi, int nomega, PerpProj p,
                                        double *__restrict__ S) {
  for (int w = blockIdx.x * blockDim.x + threadIdx.x; w < nomega; w += gridDim.x * blockDim.x) {
    double im = 0.0;
    for (int a = 0; a < 3; ++a)
      for (int b = 0; b < 3; ++b) im += p.m[a][b] * chi[((long long)a * 3 + b) * nomega + w].y;
    S[w] = -im;
  }
}

void launch_structure_factor(cudaStream_t st, const double2 *chi, int nomega, const PerpProj &p,
                             double *S) {
  structure_factor_kernel<<<blocks_for(nomega, 128), 128, 0, st>>>(chi, nomega, p, S);
  TDLZ_LAUNCH_CHECK();
}

void launch_spectrum(cudaStream_t st, const SpecArgs &a) {
  const long long nthr = (long long)a.nchain * a.nomega * a.nl;
  spectrum_kernel<<<blocks_for(nthr, kSpecThreads), kSpecThreads, 0, st>>>(a);
  TDLZ_LAUNCH_CHECK();
}

}  // namespace tdlz
