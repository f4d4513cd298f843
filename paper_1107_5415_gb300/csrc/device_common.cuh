// Device helpers shared by the transform and split kernels: complex
// arithmetic, division by run-time invariant integers, small DFT butterflies
// and reduction of integer vectors into a Hermite box.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace pfft {

// ---------------------------------------------------------------- complex
template <typename R>
struct CT;
template <>
struct CT<float> {
  using type = float2;
};
template <>
struct CT<double> {
  using type = double2;
};

// Load of data that another CTA of the same launch may have written (COH:
// through L2, bypassing the non-coherent L1 / read-only paths), or a plain
// load.
template <bool COH, typename T>
__device__ __forceinline__ T load_c(const T* p) {
  if constexpr (COH)
    return __ldcg(p);
  else
    return *p;
}

template <typename C>
__device__ __forceinline__ C cmake(decltype(C::x) a, decltype(C::x) b) {
  C c;
  c.x = a;
  c.y = b;
  return c;
}
template <typename C>
__device__ __forceinline__ C cadd(C a, C b) { return cmake<C>(a.x + b.x, a.y + b.y); }
template <typename C>
__device__ __forceinline__ C csub(C a, C b) { return cmake<C>(a.x - b.x, a.y - b.y); }
// Sums of the butterflies.  PK: one packed instruction per complex64 sum (the
// same two IEEE sums), for the kernels bound by instruction issue (M = [[512,
// 128], [0, 512]] x 16 there and back: 0.1024 -> 0.0977 ms); the pipelined row
// pass and the pipelined column pass of 1024 points, bound by their memory phases,
// keep the plain ones, which the compiler may contract with a preceding product
// (2.185 against 2.197 ms for the 2^24 x 8 step).
template <bool PK, typename C>
__device__ __forceinline__ C bsum(C a, C b) {
  if constexpr (PK && sizeof(C) == 8)
    return __fadd2_rn(a, b);
  else
    return cadd(a, b);
}
template <bool PK, typename C>
__device__ __forceinline__ C bdiff(C a, C b) {
  if constexpr (PK && sizeof(C) == 8)
    return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a);
  else
    return csub(a, b);
}
template <typename C>
__device__ __forceinline__ C cmul(C a, C b) {
  return cmake<C>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename C>
__device__ __forceinline__ C cconj(C a) { return cmake<C>(a.x, -a.y); }
// multiply by -i
template <typename C>
__device__ __forceinline__ C cmul_mi(C a) { return cmake<C>(a.y, -a.x); }
template <typename C>
__device__ __forceinline__ C cscale(C a, decltype(C::x) s) { return cmake<C>(a.x * s, a.y * s); }

// --------------------------------------------------- run-time invariant division
// Division of 0 <= n < 2^31 by a fixed divisor 1 <= d < 2^31 with one
// multiply-high, after Granlund & Montgomery, "Division by invariant integers
// using multiplication" (PLDI 1994): with l = ceil(log2 d) and
// mul = floor(2^32 (2^l - d) / d) + 1, n / d = (mulhi(n, mul) + n) >> l.
struct FastDiv {
  uint32_t d, mul, shift;
  __host__ void init(uint32_t dv) {
    d = dv;
    uint32_t l = 0;
    while ((uint64_t(1) << l) < dv) ++l;
    shift = l;
    mul = uint32_t(((uint64_t(1) << 32) * ((uint64_t(1) << l) - dv)) / dv + 1);
  }
  __device__ __forceinline__ int div(int n) const {
    uint32_t t = __umulhi(uint32_t(n), mul);
    return int((t + uint32_t(n)) >> shift);
  }
  __device__ __forceinline__ int mod(int n) const { return n - div(n) * int(d); }
};

// Quotient and remainder of 0 <= n < 2^62 by a fixed 1 <= d < 2^31, by one 64-bit
// multiply-high: mul = floor((2^64 - 1) / d) makes the estimate at most one short.
struct FastDiv64 {
  unsigned long long mul;
  uint32_t d;
  __host__ void init(uint32_t dv) {
    d = dv;
    mul = ~0ull / dv;
  }
  __device__ __forceinline__ int divmod(long long n, long long& quot) const {
    unsigned long long f = __umul64hi((unsigned long long)n, mul);
    unsigned long long r = (unsigned long long)n - f * d;
    if (r >= d) {
      r -= d;
      ++f;
    }
    quot = (long long)f;
    return int(r);
  }
  __device__ __forceinline__ int mod(long long n) const {
    long long f;
    return divmod(n, f);
  }
};

// ------------------------------------------------------------ Hermite box
// Upper-triangular H (d <= 4) with row-major slot strides.  A point y of the
// box x_r [0, H_rr) is stored as int32 coordinates.
struct BoxDesc {
  int d;
  int H[4][4];
  int stride[4];
};

// Reduce y (each coordinate in [-2 H_rr, 3 H_rr)) into the box by
// subtracting / adding columns of H, last coordinate first.
__device__ __forceinline__ void box_fix(const BoxDesc& B, int* y) {
#pragma unroll
  for (int r = 3; r >= 0; --r) {
    if (r < B.d) {
      const int h = B.H[r][r];
      while (y[r] >= h) {
        y[r] -= h;
#pragma unroll
        for (int i = 0; i < 3; ++i)
          if (i < r) y[i] -= B.H[i][r];
      }
      while (y[r] < 0) {
        y[r] += h;
#pragma unroll
        for (int i = 0; i < 3; ++i)
          if (i < r) y[i] += B.H[i][r];
      }
    }
  }
}

// Slot of reduce(a + b) for two box points a, b (tables of d int32 each).
__device__ __forceinline__ int box_sum_slot(const BoxDesc& B, const int* a, const int* b) {
  int y[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) y[r] = (r < B.d) ? a[r] + b[r] : 0;
  box_fix(B, y);
  int s = 0;
#pragma unroll
  for (int r = 0; r < 4; ++r)
    if (r < B.d) s += y[r] * B.stride[r];
  return s;
}


// Slot of reduce(a + b) for two points a, b of the box, specialised on the
// dimension.  Coordinate r of the sum lies in [0, 2 H_rr); the corrections of
// the higher coordinates shift the lower ones by at most one diagonal each,
// so every coordinate needs a bounded number of conditional steps.
template <int DIM>
__device__ __forceinline__ int box_sum_slot_t(const BoxDesc& B, const int* a, const int* b) {
  if constexpr (DIM == 1) {
    int y = a[0] + b[0];
    if (y >= B.H[0][0]) y -= B.H[0][0];
    return y;
  } else if constexpr (DIM == 2) {
    int y1 = a[1] + b[1];
    const int c1 = y1 >= B.H[1][1];
    y1 -= c1 * B.H[1][1];
    int y0 = a[0] + b[0] - c1 * B.H[0][1];
    y0 += (y0 < 0) * B.H[0][0];
    y0 -= (y0 >= B.H[0][0]) * B.H[0][0];
    return y0 * B.stride[0] + y1;
  } else if constexpr (DIM == 3) {
    int y2 = a[2] + b[2];
    const int c2 = y2 >= B.H[2][2];
    y2 -= c2 * B.H[2][2];
    int y1 = a[1] + b[1] - c2 * B.H[1][2];
    int y0 = a[0] + b[0] - c2 * B.H[0][2];
    const int c1 = (y1 >= B.H[1][1]) - (y1 < 0);
    y1 -= c1 * B.H[1][1];
    y0 -= c1 * B.H[0][1];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      y0 += (y0 < 0) * B.H[0][0];
      y0 -= (y0 >= B.H[0][0]) * B.H[0][0];
    }
    return y0 * B.stride[0] + y1 * B.stride[1] + y2;
  } else {
    return box_sum_slot(B, a, b);
  }
}

// Slot of a box point that advances by a fixed box point.  A carry out of the
// last coordinate takes H's last column off the others, so each coordinate has
// one step without and one with the carries below it; the first coordinate is
// carried in the slot itself (it wraps exactly when the slot passes m).
template <int DIM>
struct BoxWalk {
  int slot, m;
  int y1, c1, h1;          // DIM 2: last coordinate; DIM 3: middle one
  int y2, c2, h2, c1c;     // DIM 3: last coordinate; middle step with its carry
  int d0, d1, d2, d3;      // slot steps by carries (last | middle << 1)
  __device__ __forceinline__ static int wrap(int x, int n) { return x < 0 ? x + n : x >= n ? x - n : x; }
  __device__ __forceinline__ BoxWalk(const BoxDesc& B, const int* y, const int* c, int m_) : m(m_) {
    if constexpr (DIM == 1) {
      slot = y[0];
      d0 = c[0];
    } else if constexpr (DIM == 2) {
      slot = y[0] * B.stride[0] + y[1];
      y1 = y[1];
      c1 = c[1];
      h1 = B.H[1][1];
      d0 = c[0] * B.stride[0] + c1;
      d1 = wrap(c[0] - B.H[0][1], B.H[0][0]) * B.stride[0] + c1 - h1;
    } else {
      slot = y[0] * B.stride[0] + y[1] * B.stride[1] + y[2];
      y2 = y[2];
      c2 = c[2];
      h2 = B.H[2][2];
      y1 = y[1];
      c1 = c[1];
      h1 = B.H[1][1];
      const int H0 = B.H[0][0], s0 = B.stride[0], s1 = B.stride[1];
      // middle step with the carry of the last coordinate, kept in [0, h1): a
      // negative one borrows a column of its own
      const int r1 = c1 - B.H[1][2];
      c1c = r1 < 0 ? r1 + h1 : r1;
      const int x0 = wrap(c[0] - B.H[0][2], H0);                 // after the last coordinate's carry
      const int x0c = r1 < 0 ? wrap(x0 + B.H[0][1], H0) : x0;    // and the borrow
      d0 = c[0] * s0 + c1 * s1 + c2;
      d1 = x0c * s0 + c1c * s1 + c2 - h2;
      d2 = wrap(c[0] - B.H[0][1], H0) * s0 + (c1 - h1) * s1 + c2;
      d3 = wrap(x0c - B.H[0][1], H0) * s0 + (c1c - h1) * s1 + c2 - h2;
    }
  }
  __device__ __forceinline__ void step() {
    if constexpr (DIM == 1) {
      slot += d0;
    } else if constexpr (DIM == 2) {
      y1 += c1;
      const bool p = y1 >= h1;
      if (p) y1 -= h1;
      slot += p ? d1 : d0;
    } else {
      y2 += c2;
      const bool p = y2 >= h2;
      if (p) y2 -= h2;
      y1 += p ? c1c : c1;
      const bool q = y1 >= h1;
      if (q) y1 -= h1;
      const int lo = q ? d2 : d0, hi = q ? d3 : d1;
      slot += p ? hi : lo;
    }
    if (slot >= m) slot -= m;
  }
};

// A table entry of a box point: TS = 2 (d <= 2) or 4 (d = 3, 4) int32,
// fetched with one vector load.
template <int TS>
__device__ __forceinline__ void load_point(const int* __restrict__ tab, int idx, int* y) {
  if constexpr (TS == 2) {
    const int2 v = __ldg(reinterpret_cast<const int2*>(tab) + idx);
    y[0] = v.x;
    y[1] = v.y;
    y[2] = 0;
    y[3] = 0;
  } else {
    const int4 v = __ldg(reinterpret_cast<const int4*>(tab) + idx);
    y[0] = v.x;
    y[1] = v.y;
    y[2] = v.z;
    y[3] = v.w;
  }
}

// ------------------------------------------------------------- butterflies
// In-register forward DFTs, X[k] = sum_n x[n] exp(-2 pi i n k / R).
template <typename C, bool PK = true>
__device__ __forceinline__ void dft2(C& a, C& b) {
  C t = a;
  a = bsum<PK>(t, b);
  b = bdiff<PK>(t, b);
}

template <typename C, bool PK = true>
__device__ __forceinline__ void dft4(C& x0, C& x1, C& x2, C& x3) {
  C a = bsum<PK>(x0, x2), b = bdiff<PK>(x0, x2), c = bsum<PK>(x1, x3), d = cmul_mi(bdiff<PK>(x1, x3));
  x0 = bsum<PK>(a, c);
  x2 = bdiff<PK>(a, c);
  x1 = bsum<PK>(b, d);
  x3 = bdiff<PK>(b, d);
}

// exp(-2 pi i q / 16) for q = 0..15 (exact constants of cos/sin(pi/8 multiples)).
template <typename C>
__device__ __forceinline__ C w16(int q) {
  using R = decltype(C::x);
  const R c1 = R(0.92387953251128675613), s1 = R(0.38268343236508977173),
          h = R(0.70710678118654752440);
  switch (q & 15) {
    case 0: return cmake<C>(1, 0);
    case 1: return cmake<C>(c1, -s1);
    case 2: return cmake<C>(h, -h);
    case 3: return cmake<C>(s1, -c1);
    case 4: return cmake<C>(0, -1);
    case 5: return cmake<C>(-s1, -c1);
    case 6: return cmake<C>(-h, -h);
    case 7: return cmake<C>(-c1, -s1);
    case 8: return cmake<C>(-1, 0);
    case 9: return cmake<C>(-c1, s1);
    case 10: return cmake<C>(-h, h);
    case 11: return cmake<C>(-s1, c1);
    case 12: return cmake<C>(0, 1);
    case 13: return cmake<C>(s1, c1);
    case 14: return cmake<C>(h, h);
    default: return cmake<C>(c1, s1);
  }
}

// Length 8 as 4 x 2: n = 2 n1 + n2, k = k1 + 4 k2.
template <typename C, bool PK = true>
__device__ __forceinline__ void dft8(C* x) {
  C e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6];
  C o0 = x[1], o1 = x[3], o2 = x[5], o3 = x[7];
  dft4<C, PK>(e0, e1, e2, e3);
  dft4<C, PK>(o0, o1, o2, o3);
  o1 = cmul(o1, w16<C>(2));
  o2 = cmul_mi(o2);
  o3 = cmul(o3, w16<C>(6));
  x[0] = bsum<PK>(e0, o0); x[4] = bdiff<PK>(e0, o0);
  x[1] = bsum<PK>(e1, o1); x[5] = bdiff<PK>(e1, o1);
  x[2] = bsum<PK>(e2, o2); x[6] = bdiff<PK>(e2, o2);
  x[3] = bsum<PK>(e3, o3); x[7] = bdiff<PK>(e3, o3);
}

// Length 16 as 4 x 4: n = 4 n1 + n2, k = k1 + 4 k2.
template <typename C, bool PK = true>
__device__ __forceinline__ void dft16(C* x) {
  C y[16];
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) {
    C a = x[n2], b = x[4 + n2], c = x[8 + n2], d = x[12 + n2];
    dft4<C, PK>(a, b, c, d);  // over n1 -> k1
    y[n2 * 4 + 0] = a;
    y[n2 * 4 + 1] = (n2 == 0) ? b : cmul(b, w16<C>(n2));
    y[n2 * 4 + 2] = (n2 == 0) ? c : cmul(c, w16<C>(2 * n2));
    y[n2 * 4 + 3] = (n2 == 0) ? d : cmul(d, w16<C>(3 * n2));
  }
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
    C a = y[k1], b = y[4 + k1], c = y[8 + k1], d = y[12 + k1];
    dft4<C, PK>(a, b, c, d);  // over n2 -> k2
    x[k1] = a;
    x[k1 + 4] = b;
    x[k1 + 8] = c;
    x[k1 + 12] = d;
  }
}

// ---- twiddled power-of-two butterflies in fused multiply-adds (complex128: the
// double-precision pipe of two operations per clock and SM bounds those passes).
// The length-R DFT of v[r] w^r by radix-2 decimation in time, every twiddle
// factored into the odd branch of its level: the level of length len = 2^l combines
// e + T o and e - T o with T = w^(R/len) exp(-2 pi i k / len), k < len / 2, of which
// k >= len / 4 repeat k - len / 4 times -i.  e + T o takes four fused multiply-adds;
// e - T o takes four more, or two as 2 e - (e + T o), which costs a rounding: the
// last two levels of R = 16 do that, 224 operations against 268 with products by
// w .. w^15 and their powers.  The R / 2 factors T come from a table, each rounded
// once.  Relative errors (against extended precision, forward / inverse): [[1024,
// 256], [0, 1024]] 2.99e-16 / 4.20e-16, 3.07e-16 / 4.44e-16 with the powers; all levels by 2 e - s would take 192
// operations and 0.96 ms below, at up to 3% more error on small patterns.
// M = [[1024, 256], [0, 1024]] x 4, there and back: 1.222 -> 1.032 ms.
template <typename C, bool ROT, bool TWICE>
__device__ __forceinline__ void fused_butterfly(C& e, C& o, C t) {
  using Rl = decltype(C::x);
  if constexpr (ROT) t = cmul_mi(t);
  const C s = cmake<C>(fma(-t.y, o.y, fma(t.x, o.x, e.x)), fma(t.y, o.x, fma(t.x, o.y, e.y)));
  if constexpr (TWICE)
    o = cmake<C>(fma(Rl(2), e.x, -s.x), fma(Rl(2), e.y, -s.y));
  else
    o = cmake<C>(fma(t.y, o.y, fma(-t.x, o.x, e.x)), fma(-t.y, o.x, fma(-t.x, o.y, e.y)));
  e = s;
}

// Factors of level l (len = 2^l): t[fused_first(l)], k < max(1, len / 4).
__host__ __device__ constexpr int fused_first(int l) { return l <= 1 ? 0 : 1 << (l - 2); }

// R = 2 .. 16, t: the R / 2 factors
template <typename C, int R>
__device__ __forceinline__ void fused_dft(C* v, const C* t) {
  constexpr int LR = R == 16 ? 4 : R == 8 ? 3 : R == 4 ? 2 : 1;
  C a[R];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    int r = 0;
#pragma unroll
    for (int b = 0; b < LR; ++b) r |= ((i >> b) & 1) << (LR - 1 - b);
    a[i] = v[r];
  }
#pragma unroll
  for (int l = 1; l <= LR; ++l) {
    const int len = 1 << l, quarter = len / 4;
#pragma unroll
    for (int k = 0; k < (quarter ? quarter : 1); ++k) {
      const C f = t[fused_first(l) + k];
#pragma unroll
      for (int g = 0; g < R; g += len) {
        if (l <= 2) {
          fused_butterfly<C, false, false>(a[g + k], a[g + k + len / 2], f);
          if (quarter) fused_butterfly<C, true, false>(a[g + k + quarter], a[g + k + quarter + len / 2], f);
        } else {
          fused_butterfly<C, false, true>(a[g + k], a[g + k + len / 2], f);
          fused_butterfly<C, true, true>(a[g + k + quarter], a[g + k + quarter + len / 2], f);
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < R; ++i) v[i] = a[i];
}

// Any length: direct sum with roots taken from a table of omega_N^t,
// omega_R^q = tab[q * (N / R)].
template <typename C, int R>
__device__ __forceinline__ void dft_direct(C* x, const C* __restrict__ tab, int step) {
  C w[R];
#pragma unroll
  for (int q = 0; q < R; ++q) w[q] = tab[q * step];
  C y[R];
#pragma unroll
  for (int k = 0; k < R; ++k) {
    C acc = x[0];
#pragma unroll
    for (int n = 1; n < R; ++n) acc = cadd(acc, cmul(x[n], w[(n * k) % R]));
    y[k] = acc;
  }
#pragma unroll
  for (int k = 0; k < R; ++k) x[k] = y[k];
}

template <typename C, int R>
__device__ __forceinline__ void dft(C* x, const C* __restrict__ tab, int nD) {
  if constexpr (R == 2) {
    dft2(x[0], x[1]);
  } else if constexpr (R == 4) {
    dft4(x[0], x[1], x[2], x[3]);
  } else if constexpr (R == 8) {
    dft8(x);
  } else if constexpr (R == 16) {
    dft16(x);
  } else {
    dft_direct<C, R>(x, tab, nD / R);
  }
}

}  // namespace pfft
