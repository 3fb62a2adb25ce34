// FP64 X and Y line transforms of the pruned plane-wave grids on the tensor cores, by exact
// integer slices as in tc_gemm64.cuh (included by tc_gemm.cu).
//
// A line's packed side has entries at |n| <= h <= 15 only (the sphere's planes or sticks), so
// the transform of length N <= 48 is a product with a matrix of at most 31 columns (inverse) or
// rows (forward).  Folding, e_n = x_n + x_-n and o_n = x_n - x_-n, leaves a cosine and a sine
// product over n >= 0 with k >= 0,
//   X_k = E_k +- i O_k,  X_-k = E_k -+ i O_k,  E = sum_n e_n cos(2 pi n k / N), O likewise,
// for the real and the imaginary part of the line, which are two rows of the A operand: 64
// lines are 128 rows.  The line is written in fixed point, 57 bits below the power of two above
// its largest component, the matrix with 58; both as six signed digits base 1024, exact in
// FP16.  One MMA per digit i of the lines and 16 terms multiplies the matrix digits 0 .. 5 - i
// side by side into the accumulators D = i .. 5 (one MMA per pair read the lines' digits 21
// times: 2.5 ms instead of 1.4 forward below).  Every accumulator is an integer of at most 2^24
// (checked for the matrix), so that only the pairs left out, 2^-57 of the largest component, and
// the last step round.
//
// FP64 instructions bounded these passes (a warp's takes 19 clocks of an SM, and a line of 36
// some 460 of them); here none is left.  Bound by the integer instructions that split the lines
// and assemble the results (IPC 2.3).  One CTA per SM walks its share of the tiles; sixteen
// warps split and assemble, one issues the MMAs of a tile while the next one is split.  Lines
// are neighbours in memory on both sides, so that both run without staging across threads.
// Measured, X and Y passes, inverse and forward, FP64 lines -> slices, one vector: 36 x 36 x 96
// grid, 40 bands, 4 k points: 3.10 -> 1.47 and 3.09 -> 1.42 ms; 45 x 45 x 144, 24 bands, 2 k
// points: 2.71 -> 0.92 and 2.70 -> 0.88; three vectors of 24 x 24 x 48, 18 bands, 4 k points:
// 1.48 -> 1.09 and 1.47 -> 0.94.  Relative error of L x against 64-bit sums: 1.298e-16 ->
// 1.285e-16, 4.104e-16 -> 4.101e-16, 3.119e-16 -> 3.120e-16; of single lines of 12 to 48 points
// against 80-bit sums (the integer steps on the host): 4.6e-17 to 5.7e-17, an FP64 FFT's 1.1e-16
// to 2.1e-16.
#pragma once

constexpr int kLnD = 6;                        // digits
constexpr uint32_t kLnA = 128 * 16 * 2;        // bytes of one digit of the row operand, 16 terms
constexpr uint32_t kLnB = 12288;               // bytes of a direction's matrix image
constexpr unsigned long long kLnBias = 0x0802008020080200ull;  // 512 (1 + 2^10 + .. + 2^50)

// fewest tiles of one vector that take this path (not of all the stacked ones: a group's result
// is that of its sub-batches), four per CTA: 256 tiles of length 16 took 13.8 us where one thread
// per line takes 11.6.  The rule lies where slices meet the FP64 register lines (12, 16, 24, 36,
// 45); other lengths run Stockham passes below it, not measured against slices of few tiles
constexpr long long kLnMinTiles = 608;

struct LineArgs {
  const double2 *src;
  double2 *dst;
  const void *img;   // the direction's matrix digits
  const int *tab;    // entry of grid index j on the packed side, or -1 (per k; Y: per k, plane)
  const int *npl;    // Y: planes per k
  int N, h, nk, nb, npm, n3;
  int nl, st, tpr;   // lines per row, bytes between a line's elements (both sides), tiles per row
  long long sp, sf;  // row strides, packed and full side
  long long tiles;
  int *expired;      // the context's flag: a wait ran out
};

// fixed point of v, 57 bits below 2^(e - 1022)
__device__ __forceinline__ long long ln_fix(double v, int e) {
  const uint32_t hi = (uint32_t)__double2hiint(v);
  const int ex = (int)(hi >> 20) & 0x7ff;
  const uint32_t mh = (hi & 0xfffffu) | ((uint32_t)min(ex, 1) << 20);
  const unsigned long long m = ((unsigned long long)mh << 32 | (uint32_t)__double2loint(v)) << 4;
  const unsigned long long q = m >> min(e - max(ex, 1), 63);
  return (int)hi < 0 ? -(long long)q : (long long)q;
}

// FP16 pair of digit d (0: leading) of x and y, both + kLnBias: the digit's ten bits lie in two
// neighbouring bytes, at bit 0, 2, 4 or 6 of the first
__device__ __forceinline__ uint32_t ln_pair(unsigned long long x, unsigned long long y, int d) {
  const int bit = 10 * (kLnD - 1 - d), byte = bit >> 3, off = bit & 7;
  uint32_t p;
  if (byte == 3) {  // the one that crosses the words
    p = __byte_perm((uint32_t)(x >> bit), (uint32_t)(y >> bit), 0x5410);
  } else {
    const int q = byte & 3;
    p = __byte_perm(byte > 3 ? (uint32_t)(x >> 32) : (uint32_t)x,
                    byte > 3 ? (uint32_t)(y >> 32) : (uint32_t)y,
                    q | (q + 1) << 4 | (q + 4) << 8 | (q + 5) << 12) >>
        off;
  }
  p = (p & 0x03ff03ffu) | 0x64006400u;  // 1024 + digit + 512
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(p), "r"(0x66006600u));  // - 1536
  return r;
}

// sum_D f_D 1024^(4 - D), the last two rounded
__device__ __forceinline__ long long ln_sum(const int *f) {
  long long v = f[4] + ((f[5] + 512) >> 10);
  v += (long long)f[3] * (1 << 10);
  v += (long long)f[2] * (1 << 20);
  return v + (long long)(f[0] * 1024 + f[1]) * (1 << 30);
}

// v 2^(e - 1077), rounded once; out of line: zero, below 2^32, results beyond the normal range
__device__ __noinline__ double ln_value_slow(long long v, int e) {
  if (e >= 1 << 19) return __longlong_as_double(0x7ff8000000000000ll);
  if (v == 0) return 0.0;
  const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int z = __clzll((long long)a);
  const unsigned long long m = a << z;
  const double w = scalbn((double)((m >> 11) + ((m >> 10) & 1u)), e - z - 1066);
  return v < 0 ? -w : w;
}

__device__ __forceinline__ double ln_value(long long v, int e) {
  const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const uint32_t ah = (uint32_t)(a >> 32);
  const int z = __clz((int)ah), x = e + 8 - z;  // biased exponent - 1
  if (ah == 0 || (unsigned)x >= 2045u) return ln_value_slow(v, e);
  const uint32_t mh = __funnelshift_l((uint32_t)a, ah, z), ml = (uint32_t)a << z;
  // 53 bits, rounded half up; the leading one and a carry add to the exponent field
  const unsigned long long r =
      (((unsigned long long)mh << 32 | ml) >> 11) + ((ml >> 10) & 1u) +
      ((unsigned long long)((uint32_t)x << 20) << 32);
  return __hiloint2double((int)((uint32_t)(r >> 32) | ((uint32_t)(v >> 32) & 0x80000000u)),
                          (int)(uint32_t)r);
}

template <bool INV, bool Y>
__global__ void __launch_bounds__(kOzThreads, 1) line_kernel(const LineArgs g) {
  extern __shared__ __align__(1024) unsigned char tc_smem[];
  __shared__ __align__(8) uint64_t full[2], empty[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int eb[4][64];  // line exponents of the last tiles
  __shared__ int bad;
  constexpr int NI = INV ? 4 : 8;   // index pairs (n, -n) of a thread
  constexpr int kCols = INV ? 32 : 16;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nh = INV ? 1 : (g.N / 2) / 16 + 1;          // halves of n
  // A stages (inverse: two; forward: one, its results alternate between two halves of TMEM),
  // the matrix, the raw elements
  constexpr uint32_t kStage = (INV ? 2u : 4u) * kLnD * kLnA, kMat = 2u * 2u * kLnD * kLnA;
  const long long t0 = g.tiles * blockIdx.x / gridDim.x;
  const long long t1 = g.tiles * (blockIdx.x + 1) / gridDim.x;
  if (tid == 0) {
    for (int s = 0; s < 2; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&full[s])),
                   "r"(kOzSplit));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[s])));
    }
    asm volatile("fence.mbarrier_init.release.cluster;");
    bad = 0;
  }
  for (int i = tid; i < (int)(kLnB / 16); i += kOzThreads)
    reinterpret_cast<uint4 *>(tc_smem + kMat)[i] = static_cast<const uint4 *>(g.img)[i];
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_slot)),
                 "r"(512u));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_slot;
  if (warp == kOzSplit / 32) {
    // ---- MMAs of a tile once its 512 writers arrived (having read the last tile's results)
    if (lane == 0) {
      const uint32_t idesc = (1u << 4)                          // D: F32; A, B: F16
                             | ((uint32_t)(128 >> 4) << 24);    // M >> 4; N >> 3 at bit 17
      int u = 0;
      for (long long t = t0; t < t1; ++t, ++u) {
        const int s = u & 1;
        if (!mbar_wait(smem_u32(&full[s]), (uint32_t)((u >> 1) & 1))) {
          bad = 1;  // results are dropped; go on unless the stage really never came
          if (!mbar_wait_raw(smem_u32(&full[s]), (uint32_t)((u >> 1) & 1))) break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t ab = smem_u32(tc_smem) + (INV ? s * kStage : 0u);
        const uint32_t bb = smem_u32(tc_smem) + kMat, acc = tmem + (INV ? 0u : 192u * s);
        const uint64_t da0 = smem_desc(ab, 2048, 128);
        const uint64_t db0 = smem_desc(bb, kLnD * kCols * 16, 128);
        // cosine products, then sine; halves of n; both images in the order (c/s, half, digit)
        for (int q = 0; q < (INV ? 2 : 4); ++q) {
          const int cs = INV ? q : q >> 1, hh = INV ? 0 : q & 1;
          if (hh >= nh) continue;
          // digit i of the lines by digits 0 .. 5 - i of the matrix: accumulators i .. 5
#pragma unroll
          for (int i = 0; i < kLnD; ++i)
            asm volatile(
                "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
                    acc + (uint32_t)((cs * kLnD + i) * kCols)),
                "l"(da0 + (uint64_t)((q * kLnD + i) * (kLnA >> 4))),
                "l"(db0 + (uint64_t)(q * kLnD * (kCols * 32 >> 4))),
                "r"(idesc + ((uint32_t)((kLnD - i) * kCols >> 3) << 17)),
                "r"((uint32_t)(i + hh != 0)));
        }
        asm volatile(
            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                smem_u32(&empty[s])));
      }
      // the last commit covers every MMA issued: wait for it before TMEM is released
      if (u > 0) mbar_wait_raw(smem_u32(&empty[(u - 1) & 1]), (uint32_t)(((u - 1) >> 1) & 1));
    }
    __syncwarp();
  } else {
    // ---- splitting: lanes = 4 lines x (Re, Im) x 4 quarters c of n = c + 4 i; row 8 warp +
    // (lane & 7) of the operand
    const int c = lane >> 3, nmax = INV ? g.h : g.N / 2;
    const uint32_t raw = smem_u32(tc_smem) + kMat + kLnB + 8u * tid;
    // a tile's row, place in it and k, advanced tile by tile
    struct Pos {
      long long row;
      int ti, kb, k;
    };
    auto advance = [&](Pos &q) {
      if (++q.ti < g.tpr) return;
      q.ti = 0;
      ++q.row;
      if (++q.kb < 2 * g.nb) return;
      q.kb = 0;
      if (++q.k == g.nk) q.k = 0;
    };
    Pos pl, pr;  // next tile to load, next tile to write
    pl.row = t0 / g.tpr;
    pl.ti = (int)(t0 - pl.row * g.tpr);
    pl.kb = (int)(pl.row % (2 * g.nb));
    pl.k = (int)((pl.row / (2 * g.nb)) % g.nk);
    pr = pl;
    struct Line {
      long long packed, full;  // first element's offset on each side
      const int *tab;
      bool in;
    };
    auto line_at = [&](const Pos &a, int l) {
      Line q;
      const int i = a.ti * 64 + l;
      q.in = i < g.nl;
      if (Y) {
        const int p = (int)((unsigned)i / (unsigned)g.n3), j3 = i - p * g.n3;
        q.in = q.in && p < __ldg(g.npl + a.k);
        q.tab = g.tab + (a.k * g.npm + (q.in ? p : 0)) * g.N;
        q.packed = a.row * g.sp + j3;
        q.full = a.row * g.sf + p * g.N * g.n3 + j3;
      } else {
        q.tab = g.tab + a.k * g.N;
        q.packed = a.row * g.sp + i;
        q.full = a.row * g.sf + i;
      }
      return q;
    };
    auto load = [&] {
      const Line q = line_at(pl, 4 * warp + (lane & 3));
      advance(pl);
      const char *p = reinterpret_cast<const char *>(g.src + (INV ? q.packed : q.full)) +
                      ((lane & 4) << 1);
      // own element j of slot x, copied a tile ahead (zero where there is none)
      auto copy = [&](int x, int j) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(raw + 8u * kOzSplit * x),
                     "l"(p + (long long)max(j, 0) * g.st), "r"(j >= 0 ? 8 : 0)
                     : "memory");
      };
      int a[NI], b[NI];
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const int n = c + 4 * i;
        a[i] = b[i] = -1;
        if (INV) {
          if (q.in && n <= g.h) {
            a[i] = __ldg(q.tab + n);
            if (n) b[i] = __ldg(q.tab + g.N - n);
          }
        } else if (q.in && 2 * n <= g.N) {
          a[i] = n;
          if (n && 2 * n < g.N) b[i] = g.N - n;
        }
      }
      if (!q.in) p = reinterpret_cast<const char *>(g.src);
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        if (4 * i > nmax) break;
        copy(2 * i, a[i]);
        copy(2 * i + 1, b[i]);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto fetch = [&](int x) {
      double v;
      asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(raw + 8u * kOzSplit * x) : "memory");
      return v;
    };
    auto high = [&](int x) {
      int v;
      asm volatile("ld.shared.s32 %0, [%1];"
                   : "=r"(v)
                   : "r"(raw + 8u * kOzSplit * x + 4u)
                   : "memory");
      return v;
    };
    auto split = [&](int u) {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      int er = 1 << 20;
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        if (4 * i > nmax) break;
        er = max(er, max(high(2 * i) & 0x7fffffff, high(2 * i + 1) & 0x7fffffff));
      }
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) er = max(er, __shfl_xor_sync(0xffffffffu, er, o));
      er >>= 20;
      if (lane < 4) eb[u & 3][4 * warp + lane] = er;
      unsigned char *o = tc_smem + (INV ? (u & 1) * kStage : 0u) +
                         tile_off(8 * warp + (lane & 7), c >> 1, 2048) + 8 * (c & 1);
#pragma unroll
      for (int hh = 0; hh < NI / 4; ++hh) {
        if (hh >= nh) break;
        unsigned long long e[4], d[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          e[i] = d[i] = kLnBias;
          if (16 * hh + 4 * i > nmax) continue;  // no thread has such an index
          const long long a = ln_fix(fetch(8 * hh + 2 * i), er);
          const long long b = ln_fix(fetch(8 * hh + 2 * i + 1), er);
          e[i] = (unsigned long long)(a + b) + kLnBias;
          d[i] = (unsigned long long)(a - b) + kLnBias;
        }
#pragma unroll
        for (int j = 0; j < kLnD; ++j) {
          unsigned char *oj = o + (hh * kLnD + j) * kLnA;
          *reinterpret_cast<uint2 *>(oj) =
              make_uint2(ln_pair(e[0], e[1], j), ln_pair(e[2], e[3], j));
          *reinterpret_cast<uint2 *>(oj + (INV ? 1 : 2) * kLnD * kLnA) =
              make_uint2(ln_pair(d[0], d[1], j), ln_pair(d[2], d[3], j));
        }
      }
    };
    // ---- results: lane = row 32 (warp & 3) + lane, k = 4 i + (warp >> 2)
    const int quarter = warp & 3, cg = warp >> 2, part = (lane >> 2) & 1;
    const int kmax = INV ? g.N / 2 : g.h;
    const int ni = kmax >= cg ? (kmax - cg) / 4 + 1 : 0;
    const bool minus = (part == 0) == INV;  // X_k = E_k + O'_k or E_k - O'_k
    bool ok = true, dead = false;
    auto arrived = [&](int u) {
      const uint32_t at = smem_u32(&empty[u & 1]), ph = (uint32_t)((u >> 1) & 1);
      bool in = !dead && mbar_wait(at, ph);
      if (!in && !dead) dead = !mbar_wait_raw(at, ph);
      // the line exponents were written before the stage's arrivals
      if (!dead) mbar_wait_raw(smem_u32(&full[u & 1]), ph);
      ok = __all_sync(0xffffffffu, in) && ok;  // uniform: TMEM loads want whole warps
    };
    auto results = [&](int u) {
      asm volatile("tcgen05.fence::after_thread_sync;");
      const int l = 16 * quarter + (lane >> 3) * 4 + (lane & 3);
      const Line q = line_at(pr, l);
      advance(pr);
      // non-finite line, or an expired wait: beyond every range (ln_value_slow: NaN)
      const int e = eb[u & 3][l] == 0x7ff || !ok ? 1 << 20 : eb[u & 3][l];
      char *p = reinterpret_cast<char *>(g.dst + (INV ? q.full : q.packed)) + 8 * part;
      const uint32_t tb = tmem + ((uint32_t)(32 * quarter) << 16) + (INV ? 0u : 192u * (u & 1)) +
                          (uint32_t)(cg * (kCols / 4));
      auto store = [&](int j, long long x) {
        *reinterpret_cast<double *>(p + (long long)j * g.st) = ln_value(x, e);
      };
      constexpr int kStep = 2;
#pragma unroll 1
      for (int i = 0; i < ni; i += kStep) {
        uint32_t r[2][kLnD][kStep];
#pragma unroll
        for (int cs = 0; cs < 2; ++cs)
#pragma unroll
          for (int D = 0; D < kLnD; ++D)
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];"
                         : "=r"(r[cs][D][0]), "=r"(r[cs][D][1])
                         : "r"(tb + (uint32_t)((cs * kLnD + D) * kCols + i)));
        int ja[kStep], jb[kStep];  // entries of k and -k on the output side, or -1
#pragma unroll
        for (int x = 0; x < kStep; ++x) {
          const int k = 4 * (i + x) + cg;
          ja[x] = jb[x] = -1;
          if (q.in && k <= kmax) {
            ja[x] = INV ? k : __ldg(q.tab + k);
            if (k && 2 * k < g.N) jb[x] = INV ? g.N - k : __ldg(q.tab + g.N - k);
          }
        }
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int x = 0; x < kStep; ++x) {
          if (i + x >= ni) break;
          long long s[2];
#pragma unroll
          for (int a = 0; a < 2; ++a) {
            int f[kLnD];
#pragma unroll
            for (int D = 0; D < kLnD; ++D) f[D] = __float2int_rn(__uint_as_float(r[a][D][x]));
            s[a] = ln_sum(f);
          }
          long long o = __shfl_xor_sync(0xffffffffu, s[1], 4);
          if (minus) o = -o;
          if (ja[x] >= 0) store(ja[x], s[0] + o);
          if (jb[x] >= 0) store(jb[x], s[0] - o);
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;");
    };
    int u = 0;
    if (t0 < t1) load();
    for (long long t = t0; t < t1; ++t, ++u) {
      if (!INV && u > 0) arrived(u - 1);
      split(u);
      auto arrive = [&] {
        // an expired wait still arrives, so that the MMA warp and the other writers run on
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&full[u & 1]))
                     : "memory");
      };
      if (!INV) arrive();
      if (t + 1 < t1) load();
      if (u > 0) {
        if (INV) arrived(u - 1);
        results(u - 1);
      }
      if (INV) arrive();
    }
    if (u > 0) {
      arrived(u - 1);
      if (!ok) bad = 1;
      asm volatile("bar.sync 1, %0;" ::"n"(kOzSplit) : "memory");
      ok = __all_sync(0xffffffffu, ok && !bad);
      results(u - 1);
      if (!ok && lane == 0) atomicExch(g.expired, 1);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
}
