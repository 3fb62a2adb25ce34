// tdlz_spectrum_noalloc: the tridiagonal spectrum solve (continuants) for callers that
// cannot allocate device memory.  Inputs and outputs are the caller's device
// buffers; the solve keeps its state in registers (spectrum_solve.cuh).
#include <cmath>

#include "engine.cuh"
#include "spectrum_solve.cuh"

namespace tdlz {

namespace {

// One thread per (chain, omega, left vector).
__global__ void __launch_bounds__(kSpecThreads)
    spectrum_noalloc_kernel(int nchain, int nomega, int cap, const int *steps,
                            const double2 *alpha, const double *beta, const double2 *gamma,
                            const double2 *z, const double *n0, const double *wk, double start,
                            double step, double eta, int nl, double2 *chi) {
  long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (tid >= (long long)nchain * nomega * nl) return;
  const long long ciw = tid / nl;
  const int l = (int)(tid - ciw * nl);
  const int c = (int)(ciw / nomega);
  const int iw = (int)(ciw - (long long)c * nomega);
  int m = steps[c];  // read on the device: clamped to [0, cap]
  if (m > cap) m = cap;
  double2 *out = chi + ((long long)c * nl + l) * nomega + iw;
  if (m <= 0) {
    *out = make_double2(0, 0);
    return;
  }
  const double2 acc = tridiag_chi(m, alpha + (long long)c * cap, beta + (long long)c * cap,
                                  gamma + (long long)c * cap,
                                  z + ((long long)c * nl + l) * cap,
                                  make_double2(start + step * iw, eta), make_double2(0, 0));
  double s = wk[c] * n0[c];
  *out = make_double2(s * acc.x, s * acc.y);
}

}  // namespace

void spectrum_noalloc(Context &ctx, const tdlz_coeffs *c, const tdlz_spectrum_params *sp,
                      double *chi, int nomega) {
  TDLZ_REQUIRE(c && sp && chi, TDLZ_ERR_ARG, "NULL coefficients, parameters or chi");
  TDLZ_REQUIRE(c->nchain >= 1 && c->nsteps >= 1, TDLZ_ERR_ARG, "empty coefficient set");
  TDLZ_REQUIRE(c->ncomp == 0 || c->ncomp == 3 || c->ncomp == 4, TDLZ_ERR_ARG,
               "ncomp must be 0 or 3 (spin) or 4 (spin and charge)");
  TDLZ_REQUIRE(c->steps && c->alpha && c->beta && c->gamma && c->z && c->n0 && c->wk,
               TDLZ_ERR_ARG, "NULL coefficient array");
  TDLZ_REQUIRE(sp->step > 0 && sp->end >= sp->start && std::isfinite(sp->eta) && sp->eta > 0,
               TDLZ_ERR_ARG, "need step > 0, end >= start and eta > 0");
  TDLZ_REQUIRE(sp->units == 0 || sp->units == 1, TDLZ_ERR_ARG, "units must be 0 (Ha) or 1 (meV)");
  TDLZ_REQUIRE(sp->itermax0 == 0 && sp->extrapolation == 0, TDLZ_ERR_ARG,
               "tdlz_spectrum_noalloc uses every computed step and no extrapolation");
  long long nw = (long long)std::floor((sp->end - sp->start) / sp->step + 0.5) + 1;
  TDLZ_REQUIRE(nw == nomega, TDLZ_ERR_ARG,
               "nomega does not match the frequency grid (query it with tdlz_spectrum, chi = NULL)");
  TDLZ_REQUIRE(nw <= (1LL << 24), TDLZ_ERR_ARG, "at most 2^24 frequencies");
  // size limit of the interface (it dates from a form of the solve that kept four complex
  // rows per step in a static array of this many bytes)
  const long long cap_steps = ((long long)TDLZ_NOALLOC_SCRATCH_MB << 20) / 64;
  TDLZ_REQUIRE((long long)c->nsteps * c->nchain <= cap_steps, TDLZ_ERR_ARG,
               "nchain * nsteps exceeds the static scratch of tdlz_spectrum_noalloc (" +
                   std::to_string(TDLZ_NOALLOC_SCRATCH_MB) + " MiB holds nchain * nsteps <= " +
                   std::to_string(cap_steps) + ")");
  const double conv = sp->units == 1 ? 1.0 / 27211.386245988 : 1.0;
  const int nl = c->ncomp == 4 ? 4 : 3;
  spectrum_noalloc_kernel<<<blocks_for((long long)c->nchain * nomega * nl, kSpecThreads),
                            kSpecThreads, 0, ctx.stream>>>(
      c->nchain, nomega, c->nsteps, c->steps, reinterpret_cast<const double2 *>(c->alpha),
      c->beta, reinterpret_cast<const double2 *>(c->gamma),
      reinterpret_cast<const double2 *>(c->z), c->n0, c->wk, sp->start * conv, sp->step * conv,
      sp->eta * conv, nl, reinterpret_cast<double2 *>(chi));
  TDLZ_LAUNCH_CHECK();
}

}  // namespace tdlz
