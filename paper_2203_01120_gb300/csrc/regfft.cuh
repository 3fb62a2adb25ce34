// Line FFTs held entirely in one thread's registers, for lengths known at compile
// time.  The transforms are unrolled completely, so
// every array index and twiddle index is a constant: no shared memory, no
// barriers, no index arithmetic at run time.  Used for the strided x and y axes,
// where neighbouring threads own neighbouring lines and every load and store of
// a warp is coalesced without staging.
#pragma once

#include <cmath>

#include "common.cuh"

namespace tdlz {

// Twiddles of one line length, passed BY VALUE as a kernel parameter: every index
// into it is a compile-time constant after unrolling, so each twiddle is read
// straight from the kernel-parameter constant bank as an instruction operand
// (no loads, no per-device constant-memory set-up).  w[t] = exp(+2 pi i t / N).
template <class T, int N> struct RegTw {
  cx<T> w[N];
};

// Host-side table, computed once per (type, length) in double precision.
template <class T, int N> inline const RegTw<T, N> &regtw() {
  static const RegTw<T, N> tab = [] {
    RegTw<T, N> t;
    const double two_pi = 6.283185307179586476925286766559;
    for (int i = 0; i < N; ++i) {
      t.w[i].x = (T)std::cos(two_pi * i / N);
      t.w[i].y = (T)std::sin(two_pi * i / N);
    }
    return t;
  }();
  return tab;
}

// twiddle exp(+2 pi i t / N); DIR < 0 conjugates
template <class T, int DIR, int N>
__device__ __forceinline__ cx<T> rtw(const RegTw<T, N> &tw, int t) {
  cx<T> w = tw.w[t];
  if (DIR < 0) w.y = -w.y;
  return w;
}

// Complex sums, differences and real multiples s a + c of a line transform.  With PK
// (FP32) both parts go through one packed instruction: the FP32 lanes do the same work in
// half the issue slots, and half of a transform's instructions are these.
// One vector of the 36 x 36 x 96 slab (16 k points), Y + X lines in one kernel (the form before
// the slab stages), inverse / forward:
// Stockham stages 4-3-3 0.576 / 0.614 ms; this form scalar 0.593 / 0.627 ms (more registers,
// one CTA less per SM), packed with the register budget of four CTAs 0.505 / 0.587 ms.
// 45 x 45 x 144, four vectors, 8 k points: 6.38 / 6.23 -> 5.46 / 5.28 ms.  FP64 (bound by
// the FP64 pipe): 36 points 3.70 -> 3.10 ms, 45 points 3.15 -> 2.70 ms per direction.  The
// forward Z lines keep the scalar form (their packed form needs 32 registers more: 1.79
// against 1.54 ms on the 144-point lines).
template <bool PK, class V> __device__ __forceinline__ V vadd(V a, V b) {
  if constexpr (PK && sizeof(V) == 8)
    return __fadd2_rn(a, b);
  else
    return V{a.x + b.x, a.y + b.y};
}
template <bool PK, class V> __device__ __forceinline__ V vsub(V a, V b) {
  if constexpr (PK && sizeof(V) == 8)
    return __ffma2_rn(b, make_float2(-1.f, -1.f), a);  // exact: a - b rounded once
  else
    return V{a.x - b.x, a.y - b.y};
}
template <bool PK, class T, class V> __device__ __forceinline__ V vfma(T s, V a, V c) {
  if constexpr (PK && sizeof(V) == 8)
    return __ffma2_rn(make_float2(s, s), a, c);
  else
    return V{fma(s, a.x, c.x), fma(s, a.y, c.y)};
}
// c + i s d and c - i s d (s real)
template <class T>
__device__ __forceinline__ void vrot2(cx<T> c, T s, cx<T> d, cx<T> &p, cx<T> &m) {
  p = mk<T>(fma(-s, d.y, c.x), fma(s, d.x, c.y));
  m = mk<T>(fma(s, d.y, c.x), fma(-s, d.x, c.y));
}

// v * w_M^t for a compile-time t (t < M after reduction): eighths of the circle take no
// general product.
template <class T, int DIR, int M>
__device__ __forceinline__ cx<T> vtw(cx<T> v, int t, const RegTw<T, M> &tw) {
  if (t == 0) return v;
  if (2 * t == M) return mk<T>(-v.x, -v.y);
  if (4 * t == M || 4 * t == 3 * M) {
    const bool up = (4 * t == M) == (DIR > 0);
    return up ? mk<T>(-v.y, v.x) : mk<T>(v.y, -v.x);
  }
  return cmul<T>(v, rtw<T, DIR, M>(tw, t));
}

// Factor N1 of the DFT of length N = N1 N2 (0: a base butterfly).
constexpr int dft_split(int n) {
  switch (n) {
    case 2: case 3: case 4: case 5: return 0;
    case 6: return 2;
    case 8: return 2;
    case 9: return 3;
    case 10: return 2;
    case 12: return 4;
    case 15: return 3;
    case 16: return 4;
    case 18: return 2;
    case 20: return 4;
    case 24: return 8;
    case 25: return 5;
    case 27: return 3;
    case 30: return 5;
    case 32: return 4;
    case 36: return 4;
    case 40: return 8;
    case 45: return 9;
    case 48: return 16;
    default: return -1;
  }
}
constexpr int gcd_of(int a, int b) { return b == 0 ? a : gcd_of(b, a % b); }
constexpr int inv_mod(int a, int m) {  // a^-1 mod m for coprime a, m
  for (int x = 1; x < m; ++x)
    if ((a % m) * x % m == 1) return x;
  return 1;
}

// In-register DFT of length N, its roots taken from the table of a multiple M of N.
// Coprime factors (36 = 4 x 9, 45 = 9 x 5, 48 = 16 x 3, 24 = 8 x 3, ...) combine by the
// prime-factor map, which needs no twiddles between them: input n = N2 n1 + N1 n2 mod N,
// output k = k1 mod N1, k2 mod N2 (Chinese remainder).  Against the Stockham stages 4-3-3
// this leaves 16 of a 36-point line's 40 complex products with twiddles.  Other splits (8, 9, 16, 25, 27, 32) are Cooley-Tukey steps.
// All indices are compile-time constants after unrolling.
template <class T, int N, int DIR, bool PK, int M>
__device__ __forceinline__ void vdft(cx<T> (&v)[N], const RegTw<T, M> &tw) {
  if constexpr (N == 2) {
    const cx<T> a = v[0];
    v[0] = vadd<PK>(a, v[1]);
    v[1] = vsub<PK>(a, v[1]);
  } else if constexpr (N == 4) {
    const cx<T> a = vadd<PK>(v[0], v[2]), b = vsub<PK>(v[0], v[2]);
    const cx<T> c = vadd<PK>(v[1], v[3]), d = vsub<PK>(v[1], v[3]);
    v[0] = vadd<PK>(a, c);
    v[2] = vsub<PK>(a, c);
    const cx<T> p = mk<T>(b.x - d.y, b.y + d.x), m = mk<T>(b.x + d.y, b.y - d.x);
    v[1] = DIR > 0 ? p : m;
    v[3] = DIR > 0 ? m : p;
  } else if constexpr (N == 3) {
    const cx<T> w = rtw<T, DIR, M>(tw, M / 3);
    const cx<T> s = vadd<PK>(v[1], v[2]), d = vsub<PK>(v[1], v[2]);
    const cx<T> c = vfma<PK>(w.x, s, v[0]);
    v[0] = vadd<PK>(v[0], s);
    vrot2<T>(c, w.y, d, v[1], v[2]);
  } else if constexpr (N == 5) {
    const cx<T> wa = rtw<T, DIR, M>(tw, M / 5), wb = rtw<T, DIR, M>(tw, 2 * (M / 5));
    const cx<T> a1 = vadd<PK>(v[1], v[4]), b1 = vsub<PK>(v[1], v[4]);
    const cx<T> a2 = vadd<PK>(v[2], v[3]), b2 = vsub<PK>(v[2], v[3]);
    const cx<T> m1 = vfma<PK>(wb.x, a2, vfma<PK>(wa.x, a1, v[0]));
    const cx<T> m2 = vfma<PK>(wa.x, a2, vfma<PK>(wb.x, a1, v[0]));
    v[0] = vadd<PK>(v[0], vadd<PK>(a1, a2));
    cx<T> p, m;
    vrot2<T>(m1, wa.y, b1, p, m);  // m1 +- i (s1 b1 + s2 b2)
    v[1] = mk<T>(fma(-wb.y, b2.y, p.x), fma(wb.y, b2.x, p.y));
    v[4] = mk<T>(fma(wb.y, b2.y, m.x), fma(-wb.y, b2.x, m.y));
    vrot2<T>(m2, wb.y, b1, p, m);  // m2 +- i (s2 b1 - s1 b2)
    v[2] = mk<T>(fma(wa.y, b2.y, p.x), fma(-wa.y, b2.x, p.y));
    v[3] = mk<T>(fma(-wa.y, b2.y, m.x), fma(wa.y, b2.x, m.y));
  } else {
    constexpr int N1 = dft_split(N), N2 = N / N1;
    static_assert(N1 > 1 && N1 * N2 == N, "register transform length");
    constexpr bool pfa = gcd_of(N1, N2) == 1;
    cx<T> c[N1][N2];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) {
      cx<T> u[N1];
#pragma unroll
      for (int n1 = 0; n1 < N1; ++n1)
        u[n1] = v[pfa ? (N2 * n1 + N1 * n2) % N : N2 * n1 + n2];
      vdft<T, N1, DIR, PK, M>(u, tw);
#pragma unroll
      for (int k1 = 0; k1 < N1; ++k1)
        c[k1][n2] = pfa ? u[k1] : vtw<T, DIR, M>(u[k1], (k1 * n2) % N * (M / N), tw);
    }
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) {
      vdft<T, N2, DIR, PK, M>(c[k1], tw);
      constexpr int e1 = N2 * inv_mod(N2, N1), e2 = N1 * inv_mod(N1, N2);
#pragma unroll
      for (int k2 = 0; k2 < N2; ++k2)
        v[pfa ? (e1 * k1 + e2 * k2) % N : k1 + N1 * k2] = c[k1][k2];
    }
  }
}

// The register transform of a line of length N.
template <int N> struct RegPlan {
  template <class T, int DIR, bool PK = true>
  __device__ __forceinline__ static void run(cx<T> (&a)[N], const RegTw<T, N> &tw) {
    vdft<T, N, DIR, PK, N>(a, tw);
  }
};

inline bool reg_fft_length(int n) {
  return n == 12 || n == 16 || n == 24 || n == 36 || n == 45 || n == 48;
}

}  // namespace tdlz
