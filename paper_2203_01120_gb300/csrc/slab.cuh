// Plane-ordered real-space stages of the Liouvillian with stored grids (slab.cu, FP32).
#pragma once

#include "engine.cuh"

namespace tdlz {

// True when slot s can run the slab stages: square x-y grid of a register-line length,
// shared memory within the limit.
bool slab_supported(const QSlot &s);

// Slices of the partial density (a function of the slot only: it fixes the summation order).
int slab_density_chunks(const QSlot &s);

// Sticks i1t ([nvec rows][n3][nstick_max]) -> x slabs xs ([nvec rows][n3][nnp]) and, with
// density, rho[v][4][Nr] (grid order) of the nvec vectors from U slabs us and k weights.
void slab_inverse_density(Context &ctx, QSlot &s, const float2 *i1t, const float2 *us,
                          const float *wk, float2 *xs, float2 *part, float2 *rho, int nvec,
                          bool density);

// The products' coefficients pot[v][n3][3][n1 n2] from rho and v_H (grid order).
void slab_potential(Context &ctx, QSlot &s, const float2 *rho, const float2 *vh,
                    const float *fxc, const float *vloc, const float *bf, float4 *pot, int nvec,
                    bool use_h, bool use_xc);

// [v_loc + s B.sigma] x + W^s U from x slabs, U slabs and the coefficients, forward X and Y
// lines, sphere's sticks -> i1t.
void slab_product_forward(Context &ctx, QSlot &s, const float2 *xs, const float2 *us,
                          const float4 *pot, float2 *i1t, int nvec);

}  // namespace tdlz
