// FP64 contractions on the tensor cores by exact integer slices (included by tc_gemm.cu).
//
// The FP64 pipe of this part does 1.7 fused multiply-adds per clock and SM, the tensor cores
// about 3600 in FP16.  Every operand row (along the contraction) is written as fixed-point
// numbers of 62 bits below its largest exponent, and those as eight signed digits base 256:
// x = 2^(e - 1084) sum_i d_i 256^(7 - i), -128 <= d_i <= 127, exact in FP16.  A product of
// two digits has at most 2^14, so an FP32 accumulator holds the sum of the up to eight digit
// pairs (i, j) with i + j = D over 128 terms exactly (8 x 128 x 2^14 = 2^24).  Eight
// accumulators, D = 0..7 (36 of the 64 pairs; the rest lie 2^-62 below the rows' largest
// products), sit side by side in TMEM; every 128 terms they are drained into two 64-bit
// integers per output, and only the last step is FP64 (the error-free splitting of T. Ozaki,
// K. Ogita, S. Oishi, S. Rump, Numer. Algorithms 59, 2012; on integer-valued tensor-core
// sums: Mukunoki et al., ISC 2020).
//
// What is lost are bits 2^-62 below a row's largest element: nothing beside the rounding of an
// FP64 sum where the products that matter are formed by elements near the rows' largest, but
// all of it where large elements of one row meet small ones of the other (a projector that
// falls over 17 decades, a vector that grows by 10^6 over the same plane waves: 1e-12 of the
// result instead of 2e-16).  Each output is therefore tested, with quantities of its own:
// with the rows scaled by their powers of two, its error is about
//   2^-62 (||a|| + ||b|| + sqrt(K)),   K real terms,
// (truncated elements, left-out digit pairs), an FP64 sum's about 2^-53 S, S = sum |a_k| |b_k|.
// S comes from one more MMA per stage, of the two leading digits' magnitudes rounded down to
// E5M2, the norms from the pass that finds the exponents.  Where
//   S < 2^-9 (||a|| + ||b|| + sqrt(K))
// and the two rows' nonzero elements meet at all (256 bits per row, OzBits; states of opposite
// spins don't) and, in the update, the addend is as small, a second
// kernel forms the outputs of that warp's 32 x nt / 8 block by FP64 multiply-adds
// (oz_redo_kernel).  Against exact sums (the integer steps on the host, 300 to 2400 terms,
// flat, Gaussian, sparse and growing rows) outputs that pass have errors of at most
// 0.9 2^-53 S, FP64 sums of the same rows 0.7 to 8.8.
//
// One CTA per SM, with all 512 TMEM columns, walks its share of the (output tile of 128 rows x
// nt <= 48 columns, K split) list, 32 reals of K per stage, two stages: sixteen warps copy the
// next stage's operands (cp.async), split them (integer shifts and byte permutes, no FP64
// instruction) and drain the accumulators, one more issues the MMAs of a stage (issued by
// one of the splitting warps they held up the others: 12000 clocks a stage).  A row digit is
// multiplied by its 8 - i column digits side by side in one or two MMAs, so that it is read
// twice at most (one MMA per pair: 7% more time).  Tiles follow
// each other without a refill of the stages: with one CTA per tile the update's three stages
// paid start and drain each time (V_NL and P_c of 0.52 and 0.67 ms for 0.38 and 0.41).
// Bound by the split's integer instructions beside the MMAs.  Measured, FP64 pipe -> slices,
// one vector: 36 x 36 x 96 grid, 40 bands, 4 k points: V_NL 3.17 -> 0.55 ms, P_c 2.16 -> 0.57 (of
// that the rows' scales 0.07 and 0.06, the second kernels 0.01 each); 45 x 45 x 144, 24 bands, 2 k
// points: V_NL 2.25 -> 0.35, P_c 0.93 -> 0.33.  Relative error of L x against 64-bit sums:
// 1.298e-16 -> 1.284e-16 and 4.104e-16 -> 4.104e-16.
#pragma once

constexpr int kOzS = 8;                       // digits
constexpr int kOzKT = 32;                     // reals of K per stage
constexpr int kOzDrain = 4;                   // stages per drain (128 terms)
constexpr uint32_t kOzATile = 128 * kOzKT * 2;  // bytes of one digit of the row operand
constexpr int kOzMaxNt = 48;
constexpr unsigned long long kOzBias = 0x8080808080808080ull;

// biased exponent (at least 1) of |v|
__device__ __forceinline__ int oz_exp(double v) {
  return max(1, (__double2hiint(v) >> 20) & 0x7ff);
}

// digits of v below the row exponent e, as the bytes of fixed point + kOzBias (byte 7 first)
__device__ __forceinline__ unsigned long long oz_fix(double v, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int ex = (int)(b >> 52) & 0x7ff;
  unsigned long long m = b & 0xfffffffffffffull;
  if (ex) m |= 1ull << 52;
  const int s = 9 - (e - max(ex, 1));
  const unsigned long long q = s >= 0 ? m << s : s > -64 ? m >> -s : 0ull;
  return ((long long)b < 0 ? 0ull - q : q) + kOzBias;
}

// FP16 pair (digit of x, digit of y) from byte `byte` of their fixed-point words
__device__ __forceinline__ uint32_t oz_pair(unsigned long long x, unsigned long long y, int byte) {
  const uint32_t xw = byte >= 4 ? (uint32_t)(x >> 32) : (uint32_t)x;
  const uint32_t yw = byte >= 4 ? (uint32_t)(y >> 32) : (uint32_t)y;
  const int s = byte & 3;
  const uint32_t p =  // 1024 + byte of x, 1024 + byte of y
      (__byte_perm(xw, yw, s | ((4 + s) << 8)) & 0x00ff00ffu) | 0x64006400u;
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(p), "r"(0x64806480u));  // - 1152
  return r;
}

struct OzArgs {
  const double2 *A, *B;  // TN: A[a][m][k], B[b][n][k]; NN: A[b][r][k] (strided), B[g][k][n]
  long long lda, sA, ldb, sB, sar, sak;
  int amod, M, N, nj, ntot, ntm, ntn, mt, nt, nsplit, batch, kst;  // kst: stages per split
  long long K, ncol, tiles;
  const int *ea, *eb;    // exponents of A's and B's rows per split (NN: of B's columns)
  const float *na, *nb;  // their 2-norms over 2^(exponent - 1022)
  const uint4 *ba, *bb;  // which of their elements are not 0, two each (OzBits)
  float rk;              // square root of a split's real terms
  unsigned char *redo;   // [tile][16 warps]: block left to oz_redo_kernel
  double2 *part;
  const double2 *In;
  double2 *Out;
  long long ldo, sO;
  double alpha;
  int neg_from, neg_mod;
  int *expired;      // the context's flag: a wait ran out
};

// Largest biased exponent m (at least 1) of the numbers seen so far and the sum s of their
// squares over 2^(2 m - 2044), without FP64 instructions.
struct OzScale {
  int m = 1;
  float s = 0.f;
  // 2^(2 d), d <= 0; 0 below the range
  static __device__ __forceinline__ float pow4(int d) {
    return d > -63 ? __int_as_float((127 + 2 * d) << 23) : 0.f;
  }
  __device__ __forceinline__ void square(double v) {
    const uint32_t hi = (uint32_t)__double2hiint(v) & 0x7fffffffu;
    const int ex = (int)(hi >> 20), x = 126 + ex - m;
    const float f = ex > 0 && x > 0 ? __int_as_float(x << 23 | (int)((hi & 0xfffffu) << 3)) : 0.f;
    s = fmaf(f, f, s);
  }
  __device__ __forceinline__ void add(double2 v) {
    const int e = max(oz_exp(v.x), oz_exp(v.y));
    if (e > m) {
      s *= pow4(m - e);
      m = e;
    }
    square(v.x);
    square(v.y);
  }
};

// v != 0, by its words (a comparison is an FP64 instruction)
__device__ __forceinline__ bool oz_nonzero(double2 v) {
  return (((uint32_t)__double2hiint(v.x) << 1) | (uint32_t)__double2loint(v.x) |
          ((uint32_t)__double2hiint(v.y) << 1) | (uint32_t)__double2loint(v.y)) != 0;
}

// Bit of element k of a row of len: its own where len <= 256, else that of its run, 128 equal ones
// in each half (the halves of a spinor are its spins).
struct OzBits {
  uint32_t half, magic;  // of the division by the run's length
  bool own;
  __device__ OzBits(long long len) {
    own = len <= 256;
    half = (uint32_t)((len + 1) >> 1);
    magic = 0xffffffffu / ((half + 127) >> 7) + 1u;  // a run of 1: own is set
  }
  __device__ __forceinline__ int at(uint32_t k) const {
    if (own) return (int)k;
    const bool h = k >= half;
    return (int)(__umulhi(k - (h ? half : 0u), magic) + (h ? 128u : 0u));
  }
};
__device__ __forceinline__ bool oz_meet(const uint4 *a, const uint4 *b) {
  uint32_t m = 0;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const uint4 x = a[i], y = b[i];
    m |= (x.x & y.x) | (x.y & y.y) | (x.z & y.z) | (x.w & y.w);
  }
  return m != 0;
}

// exponent, norm and bits of rows of at most kc complex elements, one block per (row, split): row
// r starts at p + (r / per) s0 + (r % per) s1, elements sk apart, split y at element y kc of len
__global__ void __launch_bounds__(128)
    oz_row_scale_kernel(const double2 *__restrict__ p, int per, long long s0, long long s1,
                        long long sk, long long len, long long kc, int *__restrict__ e,
                        float *__restrict__ nrm, uint32_t *__restrict__ bits) {
  const long long r = blockIdx.x, k0 = blockIdx.y * kc, k1 = min(len, k0 + kc);
  const double2 *q = p + (r / per) * s0 + (r % per) * s1;
  const OzBits ob(len);
  const int tid = threadIdx.x;
  __shared__ int shm[4];
  __shared__ float shs[4];
  __shared__ uint32_t shb[8];
  if (tid < 8) shb[tid] = 0;
  __syncthreads();
  OzScale a;
#pragma unroll 4
  for (long long k = k0 + tid; k < k1; k += 128) {
    const double2 v = q[k * sk];
    a.add(v);
    if (oz_nonzero(v)) {
      const int b = ob.at((uint32_t)k);
      if (!(*(volatile uint32_t *)(shb + (b >> 5)) >> (b & 31) & 1u))
        atomicOr(shb + (b >> 5), 1u << (b & 31));
    }
  }
  const int wm = __reduce_max_sync(0xffffffffu, a.m);
  if ((tid & 31) == 0) shm[tid >> 5] = wm;
  __syncthreads();
  const int m = max(max(shm[0], shm[1]), max(shm[2], shm[3]));
  float s = a.s * OzScale::pow4(a.m - m);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((tid & 31) == 0) shs[tid >> 5] = s;
  __syncthreads();
  const long long at = (long long)blockIdx.y * gridDim.x + r;
  if (tid < 8) bits[8 * at + tid] = shb[tid];
  if (tid == 0) {
    e[at] = m;
    nrm[at] = sqrtf(shs[0] + shs[1] + shs[2] + shs[3]);
  }
}

// exponent, norm and bits of the columns n of B[g][k][n], k < K <= 256
__global__ void oz_col_scale_kernel(const double2 *__restrict__ B, long long ldb, long long sB,
                                    int G, int K, long long ncol, int *__restrict__ e,
                                    float *__restrict__ nrm, uint32_t *__restrict__ bits) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= G * ncol) return;
  const long long g = i / ncol;
  const double2 *q = B + g * sB + (i - g * ncol);
  OzScale a;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t m[4];
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const int k0 = 128 * h + 32 * w;
      m[w] = 0;
#pragma unroll 16
      for (int k = k0; k < min(K, k0 + 32); ++k) {
        const double2 v = q[(long long)k * ldb];
        a.add(v);
        if (oz_nonzero(v)) m[w] |= 1u << (k & 31);
      }
    }
    reinterpret_cast<uint4 *>(bits)[2 * i + h] = make_uint4(m[0], m[1], m[2], m[3]);
  }
  e[i] = a.m;
  nrm[i] = sqrtf(a.s);
}

// Magnitudes of four numbers from the FP16 pairs of their two leading digits: 256 d_0 + d_1,
// 2^14 over the row's scale, rounded down to E5M2 (the upper byte of FP16).
__device__ __forceinline__ uint32_t oz_mag(uint32_t a0, uint32_t a1, uint32_t b0, uint32_t b1) {
  uint32_t a, b;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(a) : "r"(a0), "r"(0x5c005c00u), "r"(a1));
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(b) : "r"(b0), "r"(0x5c005c00u), "r"(b1));
  return __byte_perm(a, b, 0x7531) & 0x7f7f7f7fu;
}

// Rows of the column operand's magnitudes (the S MMA's N) and bytes of a stage: digits of the
// rows, digits of the columns, magnitudes of the rows and of the columns (32 bytes a row each).
__host__ __device__ constexpr int oz_ns(int mt) { return mt > 16 ? 32 : 16; }
constexpr uint32_t kOzSTile = 128 * kOzKT;
__host__ __device__ constexpr uint32_t oz_stage(int nt, int mt) {
  return kOzS * (kOzATile + (uint32_t)nt * kOzKT * 2) + kOzSTile + (uint32_t)oz_ns(mt) * kOzKT;
}

// Tile t = ((z ntn + tn) ntm + tm): TN row tile tm of stacked (j, n), column tile tn of m,
// z = split amod + A batch; NN row tile of columns n, column tile of r, z = batch
struct OzTile {
  int tm, tn, a, sp, b, bg, nst;
  long long kc0;  // first complex k
};
template <bool NN> __device__ __forceinline__ OzTile oz_tile(const OzArgs &g, long long t) {
  OzTile q;
  q.tm = (int)(t % g.ntm);
  t /= g.ntm;
  q.tn = (int)(t % g.ntn);
  const int z = (int)(t / g.ntn);
  q.a = NN ? 0 : z % g.amod;
  q.sp = NN ? 0 : z / g.amod;
  q.b = NN ? z : 0;
  q.bg = NN ? z % g.amod : 0;  // NN: amod holds bmod
  q.kc0 = (long long)q.sp * g.kst * (kOzKT / 2);
  q.nst = (int)min((long long)g.kst, (g.K - q.kc0 + kOzKT / 2 - 1) / (kOzKT / 2));
  return q;
}
// A tile's row R: batch and index of its row operand, place of its exponent, valid or not.
struct OzRow {
  bool in;
  long long b, n, e;
};
template <bool NN>
__device__ __forceinline__ OzRow oz_row(const OzArgs &g, const OzTile &q, long long R) {
  OzRow r;
  if (NN) {
    r.in = R < g.ncol;
    r.b = q.b;
    r.n = R;
    r.e = q.bg * g.ncol + R;
  } else {
    r.in = R < g.ntot;
    const int j = (int)(R / g.N);
    r.n = R - (long long)j * g.N;
    r.b = q.a + (long long)j * g.amod;
    r.e = ((long long)q.sp * g.batch + r.b) * g.N + r.n;
  }
  return r;
}
// Place of the exponent of a tile's column cg, and of output (row, column cg).
template <bool NN>
__device__ __forceinline__ long long oz_col(const OzArgs &g, const OzTile &q, int cg) {
  return (NN ? (long long)q.b : (long long)q.sp * g.amod + q.a) * g.M + cg;
}
template <bool NN>
__device__ __forceinline__ long long oz_at(const OzArgs &g, const OzTile &q, const OzRow &r,
                                           int cg) {
  return NN ? r.b * g.sO + (long long)cg * g.ldo + r.n
            : (((long long)q.sp * g.batch + r.b) * g.M + cg) * g.N + r.n;
}

// (hi 2^32 + lo) 2^e as a double, rounded once, without an FP64 instruction
__device__ __forceinline__ double oz_value(long long hi, long long lo, int e) {
  long long h = hi + (lo >> 32);
  unsigned int l = (unsigned int)lo;  // value = h 2^32 + l
  const bool neg = h < 0;
  if (neg) {
    h = l ? ~h : -h;
    l = 0u - l;
  }
  if (h == 0 && l == 0) return 0.0;
  const int z = h ? __clzll(h) : 64 + __clz(l);
  unsigned long long m;  // the leading 64 bits
  if (z == 0)
    m = (unsigned long long)h;
  else if (z < 64)
    m = ((unsigned long long)h << z) | (z <= 32 ? (unsigned long long)l >> (32 - z)
                                                : (unsigned long long)l << (z - 32));
  else
    m = (unsigned long long)l << (z - 32);
  int x = 95 - z + e;  // exponent of the leading bit
  m = (m >> 11) + ((m >> 10) & 1u);  // 53 bits, rounded half up
  if (m >> 53) {
    m >>= 1;
    ++x;
  }
  if (x < -1022 || x > 1023) {
    const double v = scalbn((double)m, x - 52);
    return neg ? -v : v;
  }
  const unsigned long long b = ((unsigned long long)(x + 1023) << 52) | (m & 0xfffffffffffffull) |
                               (neg ? 1ull << 63 : 0ull);
  return __longlong_as_double((long long)b);
}

constexpr int kOzSplit = 512;                // threads of the splitting warps
constexpr int kOzThreads = kOzSplit + 32;   // and the MMA warp

// asynchronous 16-byte copy of a thread's own operand element into shared memory (zeros
// where `in` is false)
__device__ __forceinline__ void oz_copy(uint32_t dst, const double2 *src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
               "r"(in ? 16 : 0)
               : "memory");
}

template <bool NN>
__global__ void __launch_bounds__(kOzThreads, 1) oz_gemm_kernel(const OzArgs g) {
  extern __shared__ __align__(1024) unsigned char tc_smem[];
  __shared__ __align__(8) uint64_t full[2], empty[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int bad;  // a wait expired
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nt = g.nt;
  const uint32_t lboA = 2048, lboB = (uint32_t)(kOzS * nt) * 16;  // column digits side by side
  const uint32_t stage_bytes = oz_stage(nt, g.mt), ns = (uint32_t)oz_ns(g.mt);
  const uint32_t sOff = kOzS * (kOzATile + (uint32_t)nt * kOzKT * 2);  // magnitudes in a stage
  // tiles [t0, t1) of this CTA
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
    // ---- MMAs: stage u (counted over the CTA's tiles) holds its K tile once its 512 writers
    // arrived (after the drain of the previous accumulators, where one was due)
    if (lane == 0) {
      const uint32_t idesc = (1u << 4)                        // D: F32; A, B: F16
                             | ((uint32_t)(128 >> 4) << 24);  // M >> 4; N >> 3 at bit 17
      // magnitudes: A, B E5M2
      const uint32_t sdesc = idesc | (1u << 7) | (1u << 10) | (ns >> 3) << 17;
      int u = 0;
      bool live = true;
      for (long long t = t0; t < t1 && live; ++t) {
        const int nst = oz_tile<NN>(g, t).nst;
        for (int it = 0; it < nst; ++it, ++u) {
          const int s = u & 1;
          if (!mbar_wait(smem_u32(&full[s]), (uint32_t)((u >> 1) & 1))) {
            bad = 1;  // results are dropped; go on unless the stage really never came
            if (!mbar_wait_raw(smem_u32(&full[s]), (uint32_t)((u >> 1) & 1))) {
              live = false;
              break;
            }
          }
          asm volatile("tcgen05.fence::after_thread_sync;");
          const uint32_t ab = smem_u32(tc_smem + (size_t)s * stage_bytes);
          const uint64_t da0 = smem_desc(ab, lboA, 128);
          const uint64_t db0 = smem_desc(ab + kOzS * kOzATile, lboB, 128);
          const uint32_t ea = kOzATile >> 4;  // one digit on, in descriptors
          for (int ks = 0; ks < kOzKT / 16; ++ks) {
            const uint64_t dak = da0 + (uint64_t)(ks * (2 * lboA >> 4));
            const uint64_t dbk = db0 + (uint64_t)(ks * (2 * lboB >> 4));
            const bool fresh = (it & (kOzDrain - 1)) == 0 && ks == 0;
            // digit i of the rows by digits 0 .. 7 - i of the columns, side by side, in parts of
            // at most 256 columns: accumulators i .. 7
#pragma unroll
            for (int i = 0; i < kOzS; ++i) {
              const int all = (kOzS - i) * nt, most = 256 / nt * nt;
              for (int c0 = 0; c0 < all; c0 += most)
                asm volatile(
                    "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
                        tmem + (uint32_t)(i * nt + c0)),
                    "l"(dak + (uint64_t)(i * ea)), "l"(dbk + (uint64_t)(c0 >> 3) * 8),
                    "r"(idesc | (uint32_t)(min(most, all - c0) >> 3) << 17),
                    "r"((uint32_t)!(fresh && i == 0)));
            }
          }
          asm volatile(
              "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
              "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(
                  tmem + (uint32_t)(kOzS * nt) + ((t - t0) & 1 ? ns : 0u)),
              "l"(smem_desc(ab + sOff, 2048, 128)),
              "l"(smem_desc(ab + sOff + kOzSTile, ns * 16, 128)), "r"(sdesc), "r"((uint32_t)it));
          asm volatile(
              "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                  smem_u32(&empty[s])));
        }
      }
      // the last commit covers every MMA issued: wait for it before TMEM is released
      if (u > 0) mbar_wait_raw(smem_u32(&empty[(u - 1) & 1]), (uint32_t)(((u - 1) >> 1) & 1));
    }
    __syncwarp();
  } else {
    // ---- one row unit per thread: row tid >> 2, chunk tid & 3 (TN: 4 lanes of a row read 256
    // contiguous bytes) or row tid & 127, chunk tid >> 7 (NN: lanes read neighbouring
    // columns); one column unit (pair row tid >> 2) for the tile's first threads
    const int rrow = NN ? (tid & 127) : (tid >> 2), rch = NN ? (tid >> 7) : (tid & 3);
    const int cm = tid >> 2, cc = tid & 3;
    const double2 *rp = nullptr, *cp = nullptr;
    int re = 1, ce = 1;
    long long kc = 0;
    int nst = 0;
    auto operands = [&](long long t) {
      const OzTile q = oz_tile<NN>(g, t);
      kc = q.kc0;
      nst = q.nst;
      rp = cp = nullptr;
      re = ce = 1;
      const OzRow r = oz_row<NN>(g, q, (long long)q.tm * 128 + rrow);
      if (r.in) {
        rp = NN ? g.B + q.bg * g.sB + r.n : g.B + r.b * g.sB + r.n * g.ldb;
        re = g.eb[r.e];
      }
      const int cg = q.tn * g.mt + cm;
      if (cm < g.mt && cg < g.M) {
        cp = NN ? g.A + q.b * g.sA + (long long)cg * g.sar
                : g.A + q.a * g.sA + (long long)cg * g.lda;
        ce = g.ea[oz_col<NN>(g, q, cg)];
      }
    };
    // the thread's elements of a stage, copied a stage ahead: raw[u][thread], then the column
    // units' (threads below 4 kOzMaxNt / 2)
    constexpr int kCol = 2 * kOzMaxNt;
    const uint32_t raw = smem_u32(tc_smem) + 2 * stage_bytes;
    const uint32_t rrw = raw + 16u * tid, crw = raw + 16u * (4 * kOzSplit + tid);
    auto copy = [&](int it) {
      const long long k0 = kc + (long long)it * (kOzKT / 2);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const long long k = k0 + 4 * rch + u;
        const bool in = rp && k < g.K;
        oz_copy(rrw + 16u * kOzSplit * u, in ? (NN ? rp + k * g.ldb : rp + k) : g.B, in);
      }
      if (tid < kCol) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const long long k = k0 + 4 * cc + u;
          const bool in = cp && k < g.K;
          oz_copy(crw + 16u * kCol * u, in ? (NN ? cp + k * g.sak : cp + k) : g.A, in);
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto fetch = [](uint32_t at) {
      double2 v;
      asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(at) : "memory");
      return v;
    };
    // warp w drains lanes 32 (w & 3) .., columns (w >> 2) nt / 4 ..: nt / 4 = 4, 8 or 12
    long long hi[kOzMaxNt / 4], lo[kOzMaxNt / 4];
#pragma unroll
    for (int i = 0; i < kOzMaxNt / 4; ++i) hi[i] = lo[i] = 0;
    const int quarter = warp & 3, cq = warp >> 2, ngrp = nt >> 4;
    // the accumulators into hi (D = 0..3) and lo (D = 4..7); all MMAs on them are done
    auto drain = [&] {
      asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
      for (int q = 0; q < kOzMaxNt / 16; ++q) {
        if (q < ngrp) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t r[4][4];
#pragma unroll
            for (int D = 0; D < 4; ++D) {
              const uint32_t taddr = tmem + ((uint32_t)(32 * quarter) << 16) +
                                     (uint32_t)((4 * h + D) * nt + cq * (nt >> 2) + 4 * q);
              asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                           : "=r"(r[D][0]), "=r"(r[D][1]), "=r"(r[D][2]), "=r"(r[D][3])
                           : "r"(taddr));
            }
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              int f[4];
#pragma unroll
              for (int D = 0; D < 4; ++D) f[D] = __float2int_rn(__uint_as_float(r[D][u]));
              long long &t = h ? lo[4 * q + u] : hi[4 * q + u];
              t += ((long long)f[0] * 256 + f[1]) * 65536 + ((long long)f[2] * 256 + f[3]);
            }
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;");
    };
    // an expired wait drops the results (ok); after one that really never came, none is waited
    // for again
    bool ok = true, dead = false;
    auto arrived = [&](int s, int phase) {
      const uint32_t at = smem_u32(&empty[s]);
      bool in = !dead && mbar_wait(at, (uint32_t)(phase & 1));
      if (!in && !dead) dead = !mbar_wait_raw(at, (uint32_t)(phase & 1));
      ok = __all_sync(0xffffffffu, in) && ok;  // uniform: the drain's loads want whole warps
    };
    // outputs of a tile: row 32 quarter + lane; columns (2m, 2m + 1) = (Re, Im); sums cleared
    auto output = [&](long long t) {
      // sums of magnitudes (the next tile's are in the other half of their columns)
      float mags[kOzMaxNt / 8];
#pragma unroll
      for (int i = 0; i < kOzMaxNt / 16; ++i) {
        uint32_t r0 = 0, r1 = 0;
        if (i < ngrp)
          asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];"
                       : "=r"(r0), "=r"(r1)
                       : "r"(tmem + ((uint32_t)(32 * quarter) << 16) + kOzS * nt +
                             ((t - t0) & 1 ? ns : 0u) + (uint32_t)(cq * (nt >> 3) + 2 * i)));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        mags[2 * i] = __uint_as_float(r0);
        mags[2 * i + 1] = __uint_as_float(r1);
      }
      asm volatile("tcgen05.fence::before_thread_sync;");
      const OzTile q = oz_tile<NN>(g, t);
      const OzRow row = oz_row<NN>(g, q, (long long)q.tm * 128 + 32 * quarter + lane);
      const int m0 = q.tn * g.mt + cq * (nt >> 3);
      const int nm = min(min(nt >> 3, g.mt - cq * (nt >> 3)), g.M - m0);
      const long long c0 = oz_col<NN>(g, q, m0);
      const int er = row.in ? g.eb[row.e] : 1;
      const int *ep = g.ea + c0;
      uint32_t w = 0;  // bits c: the slices may cost column c more than FP64 rounding
      if (row.in) {
        const float lim = g.nb[row.e] + g.rk;
#pragma unroll
        for (int c = 0; c < kOzMaxNt / 8; ++c)
          if (c < nm && mags[c] < 0x1p19f * (lim + g.na[c0 + c])) w |= 1u << c;  // 2^28 2^-9
      }
      if (__any_sync(0xffffffffu, w != 0)) {
#pragma unroll
        for (int c = 0; c < kOzMaxNt / 8; ++c)
          if (w >> c & 1) {
            bool fine = !oz_meet(g.bb + 2 * row.e, g.ba + 2 * (c0 + c));
            if (NN && !fine) {
              // an addend as large as the bound takes the error with its own rounding:
              // |In / alpha| >= 2^x in units of the rows' scales, 2^(er - 1022) 2^(em - 1022)
              const double2 iv = g.In[oz_at<NN>(g, q, row, m0 + c)];
              const int x =
                  max(oz_exp(iv.x), oz_exp(iv.y)) - oz_exp(g.alpha) - (er + ep[c]) + 2043;
              const float a = __int_as_float(min(max(x + 127, 0), 254) << 23);
              fine = a >= 0x1p-9f * (g.nb[row.e] + g.rk + g.na[c0 + c]);
            }
            if (fine) w &= ~(1u << c);
          }
      }
      const bool redo = __any_sync(0xffffffffu, w != 0);
      if (lane == 0) g.redo[t * 16 + warp] = redo;
      if (row.in && !(NN && redo)) {
        const double sg = NN && (q.b % g.neg_mod) >= g.neg_from ? -1.0 : 1.0;
#pragma unroll
        for (int c = 0; c < kOzMaxNt / 8; ++c)
          if (c < nm) {
            const int em = ep[c];
            const long long at = oz_at<NN>(g, q, row, m0 + c);
            double2 v;
            v.x = oz_value(hi[2 * c], lo[2 * c], er + em - 2112);
            v.y = oz_value(hi[2 * c + 1], lo[2 * c + 1], er + em - 2112);
            if (er == 0x7ff || em == 0x7ff || !ok)  // non-finite operand, or expired wait
              v.x = v.y = __longlong_as_double(0x7ff8000000000000ll);
            if (NN) {
              const double2 iv = g.In[at];
              g.Out[at] = make_double2(sg * fma(g.alpha, v.x, iv.x), sg * fma(g.alpha, v.y, iv.y));
            } else {
              g.part[at] = v;
            }
          }
      }
#pragma unroll
      for (int i = 0; i < kOzMaxNt / 4; ++i) hi[i] = lo[i] = 0;
    };
    int u = 0;
    if (t0 < t1) {
      operands(t0);
      copy(0);
    }
    for (long long t = t0; t < t1; ++t) {
      const int n = nst;
      for (int it = 0; it < n; ++it, ++u) {
        const int s = u & 1;
        if (u >= 2) arrived(s, (u - 2) >> 1);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        unsigned char *st = tc_smem + (size_t)s * stage_bytes;
        unsigned long long x[4], y[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          const double2 v = fetch(rrw + 16u * kOzSplit * w);
          x[w] = oz_fix(v.x, re);
          y[w] = oz_fix(v.y, re);
        }
        unsigned char *o = st + tile_off(rrow, rch, lboA);
        uint4 lead;
#pragma unroll
        for (int d = 0; d < kOzS; ++d) {
          const uint4 p = make_uint4(oz_pair(x[0], y[0], 7 - d), oz_pair(x[1], y[1], 7 - d),
                                     oz_pair(x[2], y[2], 7 - d), oz_pair(x[3], y[3], 7 - d));
          *reinterpret_cast<uint4 *>(o + d * kOzATile) = p;
          if (d == 0) lead = p;
          if (d == 1)
            *reinterpret_cast<uint2 *>(st + sOff + tile_off(rrow, rch >> 1, 2048) +
                                       8 * (rch & 1)) =
                make_uint2(oz_mag(lead.x, p.x, lead.y, p.y), oz_mag(lead.z, p.z, lead.w, p.w));
        }
        if (2 * cm < nt) {
#pragma unroll
          for (int w = 0; w < 4; ++w) {
            const double2 v = fetch(crw + 16u * kCol * w);
            x[w] = oz_fix(v.x, ce);
            y[w] = oz_fix(v.y, ce);
          }
          unsigned char *oc = st + kOzS * kOzATile;
#pragma unroll
          for (int d = 0; d < kOzS; ++d) {
            uint32_t p[4], q[4], h4[4];
#pragma unroll
            for (int w = 0; w < 4; ++w) {
              // TN: Re row (x, y), Im row (-y, x); NN: Re row (x, -y), Im row (y, x)
              const uint32_t h = oz_pair(x[w], y[w], 7 - d), sw = __byte_perm(h, 0, 0x1032);
              h4[w] = h;
              p[w] = NN ? h ^ 0x80000000u : h;
              q[w] = NN ? sw : sw ^ 0x00008000u;
            }
            *reinterpret_cast<uint4 *>(oc + tile_off(d * nt + 2 * cm, cc, lboB)) =
                make_uint4(p[0], p[1], p[2], p[3]);
            *reinterpret_cast<uint4 *>(oc + tile_off(d * nt + 2 * cm + 1, cc, lboB)) =
                make_uint4(q[0], q[1], q[2], q[3]);
            if (d == 0) lead = make_uint4(h4[0], h4[1], h4[2], h4[3]);
            if (d == 1) {
              // the larger of the two parts in both places: one sum for both parts of the output
              uint2 m = make_uint2(oz_mag(lead.x, h4[0], lead.y, h4[1]),
                                   oz_mag(lead.z, h4[2], lead.w, h4[3]));
              m.x = __vmaxu4(m.x, __byte_perm(m.x, 0, 0x2301));
              m.y = __vmaxu4(m.y, __byte_perm(m.y, 0, 0x2301));
              *reinterpret_cast<uint2 *>(st + sOff + kOzSTile + tile_off(cm, cc >> 1, ns * 16) +
                                         8 * (cc & 1)) = m;
            }
          }
        }
        // this thread's elements of the next stage (its own slots: no barrier needed)
        if (it + 1 < n) {
          copy(it + 1);
        } else if (t + 1 < t1) {
          operands(t + 1);
          copy(0);
        }
        const bool due = u > 0 && (it & (kOzDrain - 1)) == 0;
        if (due) {
          // the next MMAs start the accumulators afresh: drain them first
          arrived(s ^ 1, (u - 1) >> 1);
          drain();
        }
        // an expired wait still arrives, so that the MMA warp and the other writers run on
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&full[s]))
                     : "memory");
        if (due && it == 0) output(t - 1);  // under the MMAs of the new tile
      }
    }
    if (u > 0) {
      arrived((u - 1) & 1, (u - 1) >> 1);
      if (!ok) bad = 1;
      asm volatile("bar.sync 1, %0;" ::"n"(kOzSplit) : "memory");
      ok = __all_sync(0xffffffffu, ok && !bad);
      drain();
      output(t1 - 1);
      if (!ok && lane == 0) atomicExch(g.expired, 1);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
}

// Blocks that oz_gemm_kernel left (32 rows x nt / 8 columns each) by FP64 multiply-adds: one row
// per lane, the terms in runs of eight over the four warps (a row's run is one cache line), whose
// sums are added in order.  A CTA looks through the flags of every gridDim.x-th quarter of a
// tile's rows: nothing else to do for most calls (3 us).
template <bool NN> __global__ void __launch_bounds__(128) oz_redo_kernel(const OzArgs g) {
  constexpr int kC = kOzMaxNt / 8;
  __shared__ double2 sh[4][kC][32];
  const int lane = threadIdx.x & 31, part = threadIdx.x >> 5;
  for (long long i = blockIdx.x; i < 4 * g.tiles; i += gridDim.x) {
    const long long t = i >> 2;
    const int quarter = (int)(i & 3);
    const uint4 f = *reinterpret_cast<const uint4 *>(g.redo + t * 16);
    if (((f.x | f.y | f.z | f.w) >> (8 * quarter) & 0xffu) == 0) continue;
    const OzTile q = oz_tile<NN>(g, t);
    const long long k1 = min(g.K, q.kc0 + (long long)q.nst * (kOzKT / 2));
    for (int cq = 0; cq < 4; ++cq) {
      if (!g.redo[t * 16 + 4 * cq + quarter]) continue;
      const int m0 = q.tn * g.mt + cq * (g.nt >> 3);
      const int nm = min(min(g.nt >> 3, g.mt - cq * (g.nt >> 3)), g.M - m0);
      const OzRow row = oz_row<NN>(g, q, (long long)q.tm * 128 + 32 * quarter + lane);
      double2 acc[kC];
#pragma unroll
      for (int c = 0; c < kC; ++c) acc[c] = make_double2(0.0, 0.0);
      if (row.in) {
        const double2 *bp = NN ? g.B + q.bg * g.sB + row.n : g.B + row.b * g.sB + row.n * g.ldb;
        const double2 *ap = NN ? g.A + q.b * g.sA : g.A + q.a * g.sA;
        for (long long kr = q.kc0 + 8 * part; kr < k1; kr += 32)
          for (long long k = kr; k < min(k1, kr + 8); ++k) {
            const double2 b = NN ? bp[k * g.ldb] : bp[k];
#pragma unroll
            for (int c = 0; c < kC; ++c)
              if (c < nm) {
                if (NN)
                  cfma<double>(acc[c], __ldg(ap + (m0 + c) * g.sar + k * g.sak), b);
                else
                  cfmac<double>(acc[c], __ldg(ap + (m0 + c) * g.lda + k), b);
              }
          }
      }
#pragma unroll
      for (int c = 0; c < kC; ++c) sh[part][c][lane] = acc[c];
      __syncthreads();
      for (int c = part; c < nm; c += 4)
        if (row.in) {
          double2 v = sh[0][c][lane];
          for (int i = 1; i < 4; ++i) v = cadd<double>(v, sh[i][c][lane]);
          const long long at = oz_at<NN>(g, q, row, m0 + c);
          if (NN) {
            const double2 iv = g.In[at];
            const double2 h = mk<double>(fma(g.alpha, v.x, iv.x), fma(g.alpha, v.y, iv.y));
            g.Out[at] = (q.b % g.neg_mod) >= g.neg_from ? mk<double>(-h.x, -h.y) : h;
          } else {
            g.part[at] = v;
          }
        }
      __syncthreads();
    }
  }
}
