// Plane-ordered real-space stages with stored grids (FP32, square x-y grids).
//
// After the inverse Z pass (sticks i1t[row][j3][stick]) every transform and every pointwise
// stage acts on one z plane of one band-side.  Two kernels, one CTA per (vector, z plane,
// chunk of band-sides), walk the chunk in groups of NBS band-sides:
//   inverse  sticks -> Y lines -> X lines -> x(r) slab in HBM, and in the same pass the
//            response density of the CTA's plane, summed over the chunk;
//   forward  x(r) and U slabs -> local products -> X lines -> Y lines -> sticks.
// Against the line passes with separate density and product passes, x(r) is read once
// instead of three times and written once instead of twice.  Against the plane stages
// (planes.cu), which recompute x(r) instead of storing it, each line is transformed once
// per direction, by one thread.
//
// All warps of a CTA run the phases of a group together (products, X lines, Y lines, sticks
// out; or the reverse), one line per thread in registers, and two CTAs per SM overlap their
// phases.  A first form with separate line and pointwise warps handing tiles over through
// double buffers left each side waiting for the other (14 warps, 34-37% of the issue slots:
// 9.7 and 9.2 ms for the two kernels on six vectors of the 36 x 36 x 96 slab).
//
// A tile t[row][j1 or plane][j2] of the group's 2 NBS rows sits in shared memory and is
// transformed in place: an X line owns column j2 (N entries in, the sphere's planes out, or
// the reverse), a Y line owns a plane's row.  Row pitch N + 1 keeps both directions free of
// bank conflicts.  Groups stay inside one (side, k) pair, so the sphere's tables and the
// side's signs are uniform over the CTA.
#include <algorithm>
#include <type_traits>

#include "planes.cuh"
#include "regfft.cuh"
#include "slab.cuh"

namespace tdlz {

namespace {

// Band-sides per group: the X lines of a group (2 NBS N) about fill the CTA, and two CTAs'
// tiles and stick rows fit an SM.
template <int N> struct Slab {
  static constexpr int NBS = N >= 45 ? 2 : N == 36 ? 3 : 4;
  // threads of the forward and of the inverse kernel: at 45 points and above the inverse
  // keeps six warps of up to 168 registers (line and density sums), the forward takes
  // eight of 128 for its products (45 x 45 x 144, four vectors: inverse 8.6 ms against 9.4
  // with eight warps, forward 8.7 ms against 9.4 with six)
  static constexpr int FTH = N <= 12 ? 96 : N <= 16 ? 128 : N <= 24 ? 192 : 256;
  static constexpr int ITH = N >= 45 ? 192 : FTH;
  static constexpr int CTAS = N >= 24 ? 2 : 4;  // three of 24 points spill: 0.33 for 0.21 ms
  static constexpr int PU = N >= 45 ? 4 : 2;    // points a forward thread loads at a time
  static constexpr int P = N + 1;                           // row pitch of a tile
  static constexpr int TROW = N * P;                        // elements of one row's tile
  static constexpr int TILE = 2 * NBS * TROW;
  static constexpr int NP = (N * N + ITH - 1) / ITH;  // density points per thread
  static_assert(2 * NBS * N <= ITH, "one X line per thread");
};

__device__ __forceinline__ void cp_async8(void *dst, const void *src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}

// HBM -> L2 of one contiguous plane (16-byte aligned, bytes a multiple of 16)
__device__ __forceinline__ void prefetch_l2(const void *src, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

struct SlabTab {
  const int2 *pl;   // [nk] (planes from j1 = 0 up, planes in all): the rest end at j1 = N - 1
  const int *nst;   // [nk] sticks
  const int *pos;   // [nk][nsm] stick -> plane (N + 1) + j2
  int nk, nb, n3, nsm, npm, gpp;  // gpp: groups per (side, k) pair
  long long nnp;
};

// Walks the groups [g0, g1) of a chunk: pair = side nk + k, first band of the group, and the
// pair's sphere: planes, sticks and this thread's first stick's position (read once per pair).
struct Walk {
  int pair, n, k, ns, pos0;
  int2 pl;
  __device__ Walk(const SlabTab &tb, int g, int nbs) {
    pair = g / tb.gpp;
    n = (g - pair * tb.gpp) * nbs;
    k = pair % tb.nk;
    sphere(tb);
  }
  __device__ void sphere(const SlabTab &tb) {
    ns = __ldg(tb.nst + k);
    pl = __ldg(tb.pl + k);
    pos0 = (int)threadIdx.x < ns ? __ldg(tb.pos + (long long)k * tb.nsm + threadIdx.x) : 0;
  }
  __device__ void next(const SlabTab &tb, int nbs) {
    n += nbs;
    if (n >= tb.nb) {
      n = 0;
      ++pair;
      if (++k == tb.nk) k = 0;
      if (pair < 2 * tb.nk) sphere(tb);
    }
  }
  // position of stick i = threadIdx.x + j blockDim.x
  __device__ int pos(const SlabTab &tb, int i) const {
    return i == (int)threadIdx.x ? pos0 : __ldg(tb.pos + (long long)k * tb.nsm + i);
  }
};

// ------------------------------------------------------------------ forward
// Six vectors of the 36 x 36 x 96 slab (16 k points): 5.56 ms for 20 GB of x, U and sticks
// (3.6 TB/s), against 5.32 ms (products) + 3.48 ms (X and Y lines) in two kernels; four
// vectors of 45 x 45 x 144 (8 k points): 8.7 against 8.5 + 5.3 ms.  Loads are clamped to the
// plane and the group instead of predicated (predicated ones spilled), two points per round
// (one: 6.3 ms), and the next group's planes are requested into L2 under this group's lines
// (without: 7.3 ms).
// pot[v][z][3][NN]: (w00, w11), (w01, w10), (h0, h1, B_x, -B_y) of side X; side Y exchanges
// the first two pairs' members and signs (see product).
template <int N>
__global__ void __launch_bounds__(Slab<N>::FTH, Slab<N>::CTAS)
    slab_forward_kernel(const float2 *__restrict__ xs, const float2 *__restrict__ us,
                        const float4 *__restrict__ pot, float2 *__restrict__ i1t, SlabTab tb,
                        int nvec, int glen, const RegTw<float, N> tw) {
  using D = Slab<N>;
  constexpr int NBS = D::NBS, P = D::P, NN = N * N, TH = D::FTH, PU = D::PU;
  extern __shared__ float4 slab_smem[];
  float2 *t = reinterpret_cast<float2 *>(slab_smem);  // [2 NBS][N][P]
  const int v = blockIdx.x % nvec, z = blockIdx.y;    // vectors fastest: they share U in L2
  const int g0 = blockIdx.x / nvec * glen, g1 = min(2 * tb.nk * tb.gpp, g0 + glen);
  const long long rstride = tb.n3 * tb.nnp;           // one row of a slab array
  const long long vrow = 4LL * tb.nk * tb.nb * v;
  const float4 *pp = pot + ((long long)v * tb.n3 + z) * 3 * NN;
  const int ft = threadIdx.x, xr = ft / N, xj = ft - xr * N;  // X line: row xr, column xj
  Walk wk(tb, g0, NBS);
  for (int g = g0; g < g1; ++g, wk.next(tb, NBS)) {
    const int nbg = min(NBS, tb.nb - wk.n), rows = 2 * nbg;
    const long long row0 = 2LL * ((long long)wk.pair * tb.nb + wk.n);
    // the next group's x and U planes on their way to L2 under this group's lines
    if (ft < 4 * NBS && g + 1 < g1) {
      const int r = ft >> 1;  // rows follow on, within the pair or into the next one
      const long long nr = row0 + rows + r;
      if (nr < 4LL * tb.nk * tb.nb)
        prefetch_l2((ft & 1 ? us + nr * rstride : xs + (vrow + nr) * rstride) +
                        (long long)z * tb.nnp,
                    (unsigned)(tb.nnp * sizeof(float2)));
    }
    {
      const float2 *xp = xs + (vrow + row0) * rstride + (long long)z * tb.nnp;
      const float2 *up = us + row0 * rstride + (long long)z * tb.nnp;
      // t0 = h0 x0 + (bx - i by) x1 + w00 u0 + w01 u1, t1 = h1 x1 + (bx + i by) x0 + w10 u0 +
      // w11 u1; on side Y h0 <-> h1, w00 <-> w11, and b, w01, w10 change sign
      auto product = [&](auto side_y) {
        constexpr bool Y = decltype(side_y)::value;
        // PU points per thread and round: their loads are all in flight together
        for (unsigned e0 = ft; e0 < NN; e0 += PU * TH) {
          float4 c0[PU], c1[PU], c2[PU];
          float2 x0[PU][NBS], x1[PU][NBS], u0[PU][NBS], u1[PU][NBS];
#pragma unroll
          for (int w = 0; w < PU; ++w) {
            const unsigned e = min(e0 + w * TH, (unsigned)NN - 1);
#pragma unroll
            for (int q = 0; q < NBS; ++q) {
              const long long ro = (q < nbg ? 2 * q : 0) * rstride;
              x0[w][q] = __ldcs(xp + ro + e);
              x1[w][q] = __ldcs(xp + ro + rstride + e);
              u0[w][q] = __ldg(up + ro + e);
              u1[w][q] = __ldg(up + ro + rstride + e);
            }
            c0[w] = __ldg(pp + e);
            c1[w] = __ldg(pp + NN + e);
            c2[w] = __ldg(pp + 2 * NN + e);
          }
#pragma unroll
          for (int w = 0; w < PU; ++w) {
            const unsigned e = e0 + w * TH;
            if (e < NN) {
              const float2 wa = make_float2(c0[w].x, c0[w].y), wb = make_float2(c0[w].z, c0[w].w);
              const float2 w00 = Y ? wb : wa, w11 = Y ? wa : wb;
              const float2 w01 = Y ? make_float2(-c1[w].x, -c1[w].y) : make_float2(c1[w].x, c1[w].y);
              const float2 w10 = Y ? make_float2(-c1[w].z, -c1[w].w) : make_float2(c1[w].z, c1[w].w);
              const float h0 = Y ? c2[w].y : c2[w].x, h1 = Y ? c2[w].x : c2[w].y;
              const float2 b = Y ? make_float2(-c2[w].z, -c2[w].w) : make_float2(c2[w].z, c2[w].w);
              float2 *tp = t + e / N * P + e % N;
#pragma unroll
              for (int q = 0; q < NBS; ++q)
                if (q < nbg) {
                  float2 t0 = cscale<float>(x0[w][q], h0), t1 = cscale<float>(x1[w][q], h1);
                  cfma<float>(t0, b, x1[w][q]);
                  cfma<float>(t0, w00, u0[w][q]);
                  cfma<float>(t0, w01, u1[w][q]);
                  cfma<float>(t1, make_float2(b.x, -b.y), x0[w][q]);
                  cfma<float>(t1, w10, u0[w][q]);
                  cfma<float>(t1, w11, u1[w][q]);
                  tp[2 * q * D::TROW] = t0;
                  tp[(2 * q + 1) * D::TROW] = t1;
                }
            }
          }
        }
      };
      if (wk.pair < tb.nk)
        product(std::false_type{});
      else
        product(std::true_type{});
    }
    __syncthreads();
    const int2 pl = wk.pl;
    if (xr < rows) {
      float2 *c = t + xr * D::TROW + xj;
      float2 a[N];
#pragma unroll
      for (int j = 0; j < N; ++j) a[j] = c[j * P];
      RegPlan<N>::template run<float, -1>(a, tw);
      float2 *cu = c - (N - pl.y) * P;  // planes counted from the far end
      const int hi = N - (pl.y - pl.x);
#pragma unroll
      for (int j = 0; j < N; ++j) {
        if (j < pl.x) c[j * P] = a[j];
        if (j >= hi) cu[j * P] = a[j];
      }
    }
    __syncthreads();
    for (int l = ft; l < rows * pl.y; l += TH) {
      const int r = l / pl.y, p = l - r * pl.y;
      float2 *c = t + r * D::TROW + p * P;
      float2 a[N];
#pragma unroll
      for (int j = 0; j < N; ++j) a[j] = c[j];
      RegPlan<N>::template run<float, -1>(a, tw);
#pragma unroll
      for (int j = 0; j < N; ++j) c[j] = a[j];
    }
    __syncthreads();
    {
      float2 *o = i1t + ((vrow + row0) * tb.n3 + z) * tb.nsm;
      for (int i = ft; i < wk.ns; i += TH) {
        const float2 *c = t + wk.pos(tb, i);
#pragma unroll
        for (int r = 0; r < 2 * NBS; ++r)
          if (r < rows) o[(long long)r * tb.n3 * tb.nsm + i] = c[r * D::TROW];
      }
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ inverse
// Six vectors of the slab: 5.25 ms, against 2.98 ms (Y and X lines) + 3.40 ms (density) in
// two kernels that wrote x(r) and read it back; 45 x 45 x 144 as above: 8.6 against
// 5.5 + 5.1 ms.
// Dense stick rows d[2 NBS][npm][P] (zeros where a plane has no stick) follow the tile; the
// next group's sticks are copied into them (cp.async) while this group's X lines run.
template <int N, bool DENS>
__global__ void __launch_bounds__(Slab<N>::ITH, Slab<N>::CTAS)
    slab_inverse_kernel(const float2 *__restrict__ i1t, const float2 *__restrict__ us,
                        const float *__restrict__ wk_, float2 *__restrict__ xs,
                        float2 *__restrict__ part, SlabTab tb, int nvec, int glen,
                        const RegTw<float, N> tw) {
  using D = Slab<N>;
  constexpr int NBS = D::NBS, P = D::P, NN = N * N, NP = D::NP, TH = D::ITH;
  extern __shared__ float4 slab_smem[];
  float2 *t = reinterpret_cast<float2 *>(slab_smem);  // [2 NBS][N][P]
  float2 *d = t + D::TILE;
  const int drow = tb.npm * P;
  const int v = blockIdx.x % nvec, ch = blockIdx.x / nvec, z = blockIdx.y;
  const int g0 = ch * glen, g1 = min(2 * tb.nk * tb.gpp, g0 + glen);
  const long long rstride = tb.n3 * tb.nnp;
  const long long vrow = 4LL * tb.nk * tb.nb * v;
  const int ft = threadIdx.x, xr = ft / N, xj = ft - xr * N;
  // density: n[s][s'] = sum w conj(U_s) x_s' at point e = ft + i TH.  On the Y side n00 and
  // n11 change places and n01, n10 their sign (t = 1, -1, -1, -1), so one set of sums
  // serves both sides.
  float2 n00[DENS ? NP : 1], n01[DENS ? NP : 1], n10[DENS ? NP : 1], n11[DENS ? NP : 1];
  if constexpr (DENS) {
#pragma unroll
    for (int i = 0; i < NP; ++i) n00[i] = n01[i] = n10[i] = n11[i] = make_float2(0.f, 0.f);
  }
  auto other_side = [&] {
    if constexpr (DENS) {
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        const float2 a = n00[i];
        n00[i] = n11[i];
        n11[i] = a;
        n01[i] = make_float2(-n01[i].x, -n01[i].y);
        n10[i] = make_float2(-n10[i].x, -n10[i].y);
      }
    }
  };
  auto stage = [&](const Walk &w) {
    const int rows = 2 * min(NBS, tb.nb - w.n);
    const long long row0 = vrow + 2LL * ((long long)w.pair * tb.nb + w.n);
    const float2 *src = i1t + (row0 * tb.n3 + z) * tb.nsm;
    for (int i = ft; i < w.ns; i += TH) {
      float2 *o = d + w.pos(tb, i);
#pragma unroll
      for (int r = 0; r < 2 * NBS; ++r)
        if (r < rows) cp_async8(o + r * drow, src + (long long)r * tb.n3 * tb.nsm + i);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  auto clear = [&] {
    for (int i = ft; i < 2 * NBS * drow; i += TH) d[i] = make_float2(0.f, 0.f);
    __syncthreads();
  };
  Walk wk(tb, g0, NBS);
  bool up = wk.pair < tb.nk;
  clear();
  stage(wk);
  for (int g = g0; g < g1; ++g) {
    const int nbg = min(NBS, tb.nb - wk.n), rows = 2 * nbg;
    const long long row0 = 2LL * ((long long)wk.pair * tb.nb + wk.n);
    const float wt = DENS ? __ldg(wk_ + wk.k) : 0.f;
    const int2 pl = wk.pl;
    if (DENS && up && wk.pair >= tb.nk) {
      other_side();
      up = false;
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();  // sticks landed; the tile's last readers are done
    for (int l = ft; l < rows * pl.y; l += TH) {
      const int r = l / pl.y, p = l - r * pl.y;
      const float2 *s = d + r * drow + p * P;
      float2 a[N];
#pragma unroll
      for (int j = 0; j < N; ++j) a[j] = s[j];
      RegPlan<N>::template run<float, +1>(a, tw);
      float2 *c = t + r * D::TROW + p * P;
#pragma unroll
      for (int j = 0; j < N; ++j) c[j] = a[j];
    }
    __syncthreads();
    const int pair = wk.pair;
    wk.next(tb, NBS);
    if (DENS && ft < 2 * NBS && g + 1 < g1) {  // the next group's U planes to L2
      const long long nr = row0 + rows + ft;
      if (nr < 4LL * tb.nk * tb.nb)
        prefetch_l2(us + nr * rstride + (long long)z * tb.nnp,
                    (unsigned)(tb.nnp * sizeof(float2)));
    }
    if (g + 1 < g1) {
      if (wk.pair != pair) clear();  // another sphere: its empty entries are zero again
      stage(wk);
    }
    if (xr < rows) {
      float2 *c = t + xr * D::TROW + xj;
      const float2 *cu = c - (N - pl.y) * P;
      const int hi = N - (pl.y - pl.x);
      float2 a[N];
#pragma unroll
      for (int j = 0; j < N; ++j) {
        a[j] = make_float2(0.f, 0.f);
        if (j < pl.x) a[j] = c[j * P];
        if (j >= hi) a[j] = cu[j * P];
      }
      RegPlan<N>::template run<float, +1>(a, tw);
#pragma unroll
      for (int j = 0; j < N; ++j) c[j * P] = a[j];
    }
    float2 *xp = xs + (vrow + row0) * rstride + (long long)z * tb.nnp;
    const float2 *u = us + row0 * rstride + (long long)z * tb.nnp;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const unsigned e = min(ft + i * TH, NN - 1);
      const bool own = ft + i * TH < NN;
      const float2 *tp = t + e / N * P + e % N;
      float2 u0[NBS], u1[NBS];
      if constexpr (DENS) {
#pragma unroll
        for (int q = 0; q < NBS; ++q) {
          const long long ro = (q < nbg ? 2 * q : 0) * rstride;
          u0[q] = __ldg(u + ro + e);
          u1[q] = __ldg(u + ro + rstride + e);
        }
      }
#pragma unroll
      for (int q = 0; q < NBS; ++q) {
        // bands beyond the group read its first rows at zero weight
        const int tq = q < nbg ? 2 * q * D::TROW : 0;
        const float2 x0 = tp[tq], x1 = tp[tq + D::TROW];
        if (own && q < nbg) {
          xp[2 * q * rstride + e] = x0;
          xp[(2 * q + 1) * rstride + e] = x1;
        }
        if constexpr (DENS) {
          const float wq = q < nbg ? wt : 0.f;
          const float2 a0 = cscale<float>(u0[q], wq), a1 = cscale<float>(u1[q], wq);
          cfmac<float>(n00[i], a0, x0);
          cfmac<float>(n01[i], a0, x1);
          cfmac<float>(n10[i], a1, x0);
          cfmac<float>(n11[i], a1, x1);
        }
      }
    }
  }
  if constexpr (DENS) {
    if (!up) other_side();
    float2 *o = part + (((long long)ch * nvec + v) * 4 * tb.n3 + z) * NN;
    const long long st = (long long)tb.n3 * NN;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const int e = ft + i * TH;
      if (e >= NN) break;
      const float2 m = csub<float>(n10[i], n01[i]);  // m_y: i (n10 - n01)
      o[e] = cadd<float>(n00[i], n11[i]);
      o[st + e] = cadd<float>(n01[i], n10[i]);
      o[2 * st + e] = make_float2(-m.y, m.x);
      o[3 * st + e] = csub<float>(n00[i], n11[i]);
    }
  }
}

// rho[v][a][i n3 + j3] = sum_c part[c][v][a][j3][i] in fixed order
__global__ void slab_reduce_kernel(const float2 *__restrict__ part, float2 *__restrict__ rho,
                                   int nchunk, long long nn, int n3, long long total) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    float2 s = part[e];
    for (int c = 1; c < nchunk; ++c) s = cadd<float>(s, part[(long long)c * total + e]);
    const long long plane = nn * n3;
    const long long va = e / plane, rem = e - va * plane;
    const long long j3 = rem / nn, i = rem - j3 * nn;
    rho[va * plane + i * n3 + j3] = s;
  }
}

// v_a = delta_a0 vH + sum_b f_ab rho_b (f packed 00,01,02,03,11,12,13,22,23,33) as the
// product's coefficients of side X: w00 = v0 + v3, w11 = v0 - v3, w01 = v1 - i v2,
// w10 = v1 + i v2, h0 = vloc + B_z, h1 = vloc - B_z, (B_x, -B_y).
__global__ void slab_potential_kernel(const float2 *__restrict__ rho,
                                      const float2 *__restrict__ vh, const float *__restrict__ f,
                                      const float *__restrict__ vloc,
                                      const float *__restrict__ bf, float4 *__restrict__ pot,
                                      long long nr, int n3, int nn, int use_h, int use_xc) {
  rho += blockIdx.y * 4LL * nr;
  vh += blockIdx.y * nr;
  pot += blockIdx.y * 3LL * nr;
  for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < nr;
       r += (long long)gridDim.x * blockDim.x) {
    float2 v[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) v[a] = make_float2(0.f, 0.f);
    if (use_xc) {
      float2 p[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) p[a] = rho[a * nr + r];
      int q = 0;
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = a; b < 4; ++b) {
          const float fv = f[q++ * nr + r];
          v[a] = make_float2(fmaf(fv, p[b].x, v[a].x), fmaf(fv, p[b].y, v[a].y));
          if (b != a) v[b] = make_float2(fmaf(fv, p[a].x, v[b].x), fmaf(fv, p[a].y, v[b].y));
        }
    }
    if (use_h) v[0] = cadd<float>(v[0], vh[r]);
    const float vl = vloc[r], bx = bf[r], by = bf[nr + r], bz = bf[2 * nr + r];
    const long long i = r / n3, j3 = r - i * n3;
    float4 *o = pot + j3 * 3 * nn + i;
    o[0] = make_float4(v[0].x + v[3].x, v[0].y + v[3].y, v[0].x - v[3].x, v[0].y - v[3].y);
    o[nn] = make_float4(v[1].x + v[2].y, v[1].y - v[2].x, v[1].x - v[2].y, v[1].y + v[2].x);
    o[2 * nn] = make_float4(vl + bz, vl - bz, bx, -by);
  }
}

constexpr size_t kSlabSmem = 227 * 1024;

template <int N> size_t smem_fwd() { return (size_t)Slab<N>::TILE * sizeof(float2); }
template <int N> size_t smem_inv(int npm) {
  return smem_fwd<N>() + (size_t)2 * Slab<N>::NBS * npm * Slab<N>::P * sizeof(float2);
}

#define TDLZ_SLAB_SWITCH(n, CALL)       \
  switch (n) {                          \
    case 12: CALL(12); break;           \
    case 16: CALL(16); break;           \
    case 24: CALL(24); break;           \
    case 36: CALL(36); break;           \
    case 45: CALL(45); break;           \
    case 48: CALL(48); break;           \
    default: TDLZ_REQUIRE(false, TDLZ_ERR_STATE, "slab stages: unsupported grid length"); \
  }

int nbs_of(int n) { return n >= 45 ? 2 : n == 36 ? 3 : 4; }

SlabTab tab_of(const QSlot &s) {
  SlabTab t;
  t.pl = s.slab_pl.as<int2>();
  t.nst = s.st_n.as<int>();
  t.pos = s.slab_pos.as<int>();
  t.nk = s.nk;
  t.nb = s.nb;
  t.n3 = s.fft[2];
  t.nsm = s.nstick_max;
  t.npm = s.slab_npm;
  t.gpp = (s.nb + nbs_of(s.fft[0]) - 1) / nbs_of(s.fft[0]);
  t.nnp = planes_nnp(s);
  return t;
}

// Groups per CTA for about `ctas` CTAs over nvec vectors and every z plane; at least four
// where there are that many.
int group_len(const QSlot &s, int nvec, long long ctas) {
  const int q = nbs_of(s.fft[0]), ngrp = 2 * s.nk * ((s.nb + q - 1) / q);
  const long long base = (long long)nvec * s.fft[2], want = (ctas + base - 1) / base;
  const long long n = std::max(1LL, std::min(want, (long long)(ngrp + 3) / 4));
  return (int)((ngrp + n - 1) / n);
}
// a function of the slot only (one vector's waves): it fixes the density's summation order
int density_len(const QSlot &s) { return group_len(s, 1, 10LL * 304); }
int groups_of(const QSlot &s) {
  const int q = nbs_of(s.fft[0]);
  return 2 * s.nk * ((s.nb + q - 1) / q);
}

}  // namespace

bool slab_supported(const QSlot &s) {
  const int n = s.fft[0];
  if (s.fft[1] != n || !reg_fft_length(n)) return false;
  size_t sm = kSlabSmem + 1;
  switch (n) {
    case 12: sm = smem_inv<12>(s.slab_npm); break;
    case 16: sm = smem_inv<16>(s.slab_npm); break;
    case 24: sm = smem_inv<24>(s.slab_npm); break;
    case 36: sm = smem_inv<36>(s.slab_npm); break;
    case 45: sm = smem_inv<45>(s.slab_npm); break;
    case 48: sm = smem_inv<48>(s.slab_npm); break;
    default: break;
  }
  return sm <= kSlabSmem && s.fft[2] <= 65535;
}

int slab_density_chunks(const QSlot &s) {
  const int len = density_len(s);
  return (groups_of(s) + len - 1) / len;
}

void slab_inverse_density(Context &ctx, QSlot &s, const float2 *i1t, const float2 *us,
                          const float *wk, float2 *xs, float2 *part, float2 *rho, int nvec,
                          bool density) {
  const int len = density_len(s), nch = (groups_of(s) + len - 1) / len;
  const dim3 grid((unsigned)(nvec * nch), (unsigned)s.fft[2]);
#define TDLZ_SLAB_INV(NV)                                                                     \
  {                                                                                           \
    const size_t sm = smem_inv<NV>(s.slab_npm);                                             \
    auto kern = density ? slab_inverse_kernel<NV, true> : slab_inverse_kernel<NV, false>;     \
    TDLZ_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm)); \
    kern<<<grid, Slab<NV>::ITH, sm, ctx.stream>>>(i1t, us, wk, xs, part, tab_of(s), nvec,  \
                                                  len, regtw<float, NV>());               \
  }
  TDLZ_SLAB_SWITCH(s.fft[0], TDLZ_SLAB_INV)
#undef TDLZ_SLAB_INV
  TDLZ_LAUNCH_CHECK();
  if (!density) return;
  const long long total = (long long)nvec * 4 * s.nr;
  slab_reduce_kernel<<<blocks_for(total), 256, 0, ctx.stream>>>(
      part, rho, nch, (long long)s.fft[0] * s.fft[1], s.fft[2], total);
  TDLZ_LAUNCH_CHECK();
}

void slab_potential(Context &ctx, QSlot &s, const float2 *rho, const float2 *vh,
                    const float *fxc, const float *vloc, const float *bf, float4 *pot, int nvec,
                    bool use_h, bool use_xc) {
  const int th = spread_threads(s.nr, nvec);
  slab_potential_kernel<<<dim3(blocks_for(s.nr, th), nvec), th, 0, ctx.stream>>>(
      rho, vh, fxc, vloc, bf, pot, s.nr, s.fft[2], s.fft[0] * s.fft[1], use_h ? 1 : 0,
      use_xc ? 1 : 0);
  TDLZ_LAUNCH_CHECK();
}

void slab_product_forward(Context &ctx, QSlot &s, const float2 *xs, const float2 *us,
                          const float4 *pot, float2 *i1t, int nvec) {
  const int len = group_len(s, nvec, 10LL * 304);
  const dim3 grid((unsigned)(nvec * ((groups_of(s) + len - 1) / len)), (unsigned)s.fft[2]);
#define TDLZ_SLAB_FWD(NV)                                                                     \
  {                                                                                           \
    const size_t sm = smem_fwd<NV>();                                                         \
    auto kern = slab_forward_kernel<NV>;                                                      \
    TDLZ_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm)); \
    kern<<<grid, Slab<NV>::FTH, sm, ctx.stream>>>(xs, us, pot, i1t, tab_of(s), nvec, len,  \
                                                      regtw<float, NV>());                    \
  }
  TDLZ_SLAB_SWITCH(s.fft[0], TDLZ_SLAB_FWD)
#undef TDLZ_SLAB_FWD
  TDLZ_LAUNCH_CHECK();
}

}  // namespace tdlz
