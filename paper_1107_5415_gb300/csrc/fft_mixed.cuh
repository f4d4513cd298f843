// Mixed-radix passes of the Kronecker factorisation (Theorem 1, eq.
// (KroneckerFFT)) for any cycle lengths: row tiles, column tiles and tiles
// that hold whole signals (fft_mixed.hpp), each a batched Stockham autosort DFT
// in shared memory with the exact gather / scatter between the Hermite boxes
// and the Smith coordinates fused into its global loads and stores.
//
// What bounds these passes is the issue of instructions, not the memory: a
// stage costs a point about 28 of them whatever its radix (shared-memory round
// trip, addresses, butterfly, twiddles), so the planner covers a cycle with the
// fewest stages out of the radices up to 16 (10800 = 16 15 15 3), composite
// radices run as one register butterfly (Good's prime-factor index map, no
// inner twiddles), and complex64 sums and real multiples are packed
// instructions.  A thread holds at most 16 points and 64 registers, so 1024
// threads are resident per SM, in one tile or several.
//
// There and back (forward and inverse), in one shared-memory kernel over radices 16,
// 8, 4, 2, 3, 5, 7 with indices from tables and here: [[1200, 240], [0, 1080]] x 8: 1.538
// and 0.39 ms (450 and 151 thread instructions a point in the row pass); [[2048, 8],
// [0, 2048]] x 8: 1.99 and 0.96 ms; [[64, 16], [-16, 64]] x 1: 88 and 25 us; a mix of
// 512 patterns, split once: 3.65 and 2.2 ms.  Reading the workspace straight into the
// first butterflies of a column tile and writing it from the last ones saves
// instructions in such tiles but costs every other stage (0.415 ms for the first), and
// so does a copy of the load and store loops without bounds checks (0.393 against
// 0.389: the instruction cache).
#pragma once
#include <cuda_runtime.h>

#include "fft_mixed.hpp"

namespace pfft {

// ------------------------------------------------------------- butterflies
// cos and sin of 2 pi q / R, q = 1 .. (R - 1) / 2, R = 3, 5, 7, 11, 13
template <int R>
__device__ __forceinline__ double odd_cos(int q) {
  if constexpr (R == 3) {
    const double t[] = {-0.5};
    return t[q - 1];
  } else if constexpr (R == 5) {
    const double t[] = {0.3090169943749474241, -0.8090169943749474241};
    return t[q - 1];
  } else if constexpr (R == 7) {
    const double t[] = {0.62348980185873353053, -0.22252093395631440429, -0.90096886790241912624};
    return t[q - 1];
  } else if constexpr (R == 11) {
    const double t[] = {0.84125353283118116886, 0.41541501300188642553, -0.14231483827328514044,
                        -0.65486073394528506406, -0.95949297361449738989};
    return t[q - 1];
  } else {
    const double t[] = {0.8854560256532098959, 0.56806474673115580251, 0.12053668025532305335,
                        -0.35460488704253562597, -0.74851074817110109863, -0.97094181742605202716};
    return t[q - 1];
  }
}
template <int R>
__device__ __forceinline__ double odd_sin(int q) {
  if constexpr (R == 3) {
    const double t[] = {0.86602540378443864676};
    return t[q - 1];
  } else if constexpr (R == 5) {
    const double t[] = {0.95105651629515357212, 0.58778525229247312917};
    return t[q - 1];
  } else if constexpr (R == 7) {
    const double t[] = {0.78183148246802980871, 0.97492791218182360702, 0.43388373911755812048};
    return t[q - 1];
  } else if constexpr (R == 11) {
    const double t[] = {0.54064081745559758211, 0.90963199535451837141, 0.98982144188093273238,
                        0.75574957435425828377, 0.28173255684142969771};
    return t[q - 1];
  } else {
    const double t[] = {0.46472317204376854566, 0.82298386589365639458, 0.9927088740980539928,
                        0.93501624268541482344, 0.66312265824079520238, 0.23931566428755776715};
    return t[q - 1];
  }
}

// acc + a s, s real
template <typename C>
__device__ __forceinline__ C cfma_r(C a, decltype(C::x) s, C acc) {
  return cmake<C>(fma(a.x, s, acc.x), fma(a.y, s, acc.y));
}
template <>
__device__ __forceinline__ float2 cfma_r(float2 a, float s, float2 acc) {
  return __ffma2_rn(a, make_float2(s, s), acc);
}

// Odd prime length in real-symmetric form: with a_m = x_m + x_{R-m} and b_m =
// x_m - x_{R-m}, y_q and y_{R-q} are t -+ i u, t = x_0 + sum a_m cos, u = sum b_m sin.
template <typename C, int R>
__device__ __forceinline__ void dft_odd(C* x) {
  using Rl = decltype(C::x);
  constexpr int h = (R - 1) / 2;
  C a[h], b[h];
  C y0 = x[0];
#pragma unroll
  for (int m = 0; m < h; ++m) {
    a[m] = bsum<true>(x[1 + m], x[R - 1 - m]);
    b[m] = bdiff<true>(x[1 + m], x[R - 1 - m]);
    y0 = bsum<true>(y0, a[m]);
  }
#pragma unroll
  for (int q = 1; q <= h; ++q) {
    C t = x[0], u;
#pragma unroll
    for (int m = 1; m <= h; ++m) {
      const int e = (q * m) % R;
      const Rl c = Rl(odd_cos<R>(e <= h ? e : R - e));
      const Rl s = e <= h ? Rl(odd_sin<R>(e)) : -Rl(odd_sin<R>(R - e));
      t = cfma_r(a[m - 1], c, t);
      u = m == 1 ? cscale(b[0], s) : cfma_r(b[m - 1], s, u);
    }
    x[q] = cmake<C>(t.x + u.y, t.y - u.x);
    x[R - q] = cmake<C>(t.x - u.y, t.y + u.x);
  }
  x[0] = y0;
}

template <typename C, int R>
__device__ __forceinline__ void mdft(C* x);

__host__ __device__ constexpr int mod_inverse(int a, int m) {
  for (int x = 1; x < m; ++x)
    if (a * x % m == 1) return x;
  return 0;
}

// Coprime factors P x Q: input n = (Q n1 + P n2) mod R, output
// k = (Q Q^-1 k1 + P P^-1 k2) mod R, a plain P x Q DFT in between (I. J. Good,
// "The interaction algorithm and practical Fourier analysis", 1958).
template <typename C, int P, int Q>
__device__ __forceinline__ void dft_coprime(C* x) {
  constexpr int R = P * Q;
  constexpr int e1 = Q * mod_inverse(Q % P, P), e2 = P * mod_inverse(P % Q, Q);
  C y[R];
#pragma unroll
  for (int n2 = 0; n2 < Q; ++n2) {
    C u[P];
#pragma unroll
    for (int n1 = 0; n1 < P; ++n1) u[n1] = x[(Q * n1 + P * n2) % R];
    mdft<C, P>(u);
#pragma unroll
    for (int k1 = 0; k1 < P; ++k1) y[k1 * Q + n2] = u[k1];
  }
#pragma unroll
  for (int k1 = 0; k1 < P; ++k1) {
    C u[Q];
#pragma unroll
    for (int n2 = 0; n2 < Q; ++n2) u[n2] = y[k1 * Q + n2];
    mdft<C, Q>(u);
#pragma unroll
    for (int k2 = 0; k2 < Q; ++k2) x[(e1 * k1 + e2 * k2) % R] = u[k2];
  }
}

// Length 9 as 3 x 3: n = 3 n1 + n2, k = k1 + 3 k2, with exp(-2 pi i n2 k1 / 9) between.
template <typename C>
__device__ __forceinline__ void dft9(C* x) {
  using Rl = decltype(C::x);
  const C w1 = cmake<C>(Rl(0.7660444431189780352), -Rl(0.64278760968653932632));
  const C w2 = cmake<C>(Rl(0.17364817766693034885), -Rl(0.98480775301220805937));
  const C w4 = cmake<C>(Rl(-0.93969262078590838405), -Rl(0.34202014332566873304));
  C y[9];
#pragma unroll
  for (int n2 = 0; n2 < 3; ++n2) {
    C u[3] = {x[n2], x[3 + n2], x[6 + n2]};
    dft_odd<C, 3>(u);
    y[n2] = u[0];
    y[3 + n2] = n2 == 0 ? u[1] : cmul(u[1], n2 == 1 ? w1 : w2);
    y[6 + n2] = n2 == 0 ? u[2] : cmul(u[2], n2 == 1 ? w2 : w4);
  }
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) {
    C u[3] = {y[3 * k1], y[3 * k1 + 1], y[3 * k1 + 2]};
    dft_odd<C, 3>(u);
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) x[k1 + 3 * k2] = u[k2];
  }
}

template <typename C, int R>
__device__ __forceinline__ void mdft(C* x) {
  if constexpr (R == 2) {
    dft2(x[0], x[1]);
  } else if constexpr (R == 4) {
    dft4(x[0], x[1], x[2], x[3]);
  } else if constexpr (R == 8) {
    dft8(x);
  } else if constexpr (R == 16) {
    dft16(x);
  } else if constexpr (R == 9) {
    dft9(x);
  } else if constexpr (R == 6) {
    dft_coprime<C, 3, 2>(x);
  } else if constexpr (R == 10) {
    dft_coprime<C, 5, 2>(x);
  } else if constexpr (R == 12) {
    dft_coprime<C, 3, 4>(x);
  } else if constexpr (R == 14) {
    dft_coprime<C, 7, 2>(x);
  } else if constexpr (R == 15) {
    dft_coprime<C, 5, 3>(x);
  } else {
    dft_odd<C, R>(x);
  }
}

// ------------------------------------------------------------------ stages
// v[r] *= w^r.  The stage table holds w^(2^b), lanes of consecutive k on
// consecutive entries; w^r = w^(r - r mod 4) w^(r mod 4) keeps three low powers
// and one high one live, and no factor carries more than log2(R) - 1 rounded
// products.
// Power-of-two radices of complex128 run as fused_dft on its R / 2 factors.
template <typename C, int R>
constexpr bool kMixFused = sizeof(C) == 16 && (R & (R - 1)) == 0;
template <typename C, int R>
constexpr int kMixPowers = kMixFused<C, R> ? R / 2 : R > 8 ? 4 : R > 4 ? 3 : R > 2 ? 2 : 1;

template <typename C, int R>
__device__ __forceinline__ void mix_twiddle(C* v, const C* w) {
  C lo[4];
  lo[1] = w[0];
  if constexpr (R > 2) lo[2] = w[1];
  if constexpr (R > 3) lo[3] = cmul(lo[1], lo[2]);
#pragma unroll
  for (int r = 1; r < R && r < 4; ++r) v[r] = cmul(v[r], lo[r]);
  if constexpr (R > 4) {
    v[4] = cmul(v[4], w[2]);
#pragma unroll
    for (int r = 5; r < R && r < 8; ++r) v[r] = cmul(v[r], cmul(w[2], lo[r - 4]));
  }
  if constexpr (R > 8) {
    v[8] = cmul(v[8], w[3]);
#pragma unroll
    for (int r = 9; r < R && r < 12; ++r) v[r] = cmul(v[r], cmul(w[3], lo[r - 8]));
  }
  if constexpr (R > 12) {
    const C w12 = cmul(w[2], w[3]);
    v[12] = cmul(v[12], w12);
#pragma unroll
    for (int r = 13; r < R; ++r) v[r] = cmul(v[r], cmul(w12, lo[r - 12]));
  }
}

template <typename C, int R>
__device__ __forceinline__ void mix_stage(C* sm, const MixDesc& a, const MixStage& s) {
  constexpr int NB = kMixPoints / R;  // butterflies a thread holds (at least one)
  constexpr int NP = kMixPowers<C, R>;
  const int total = a.n / R;
  const int istep = s.istep, ostep = s.ostep;
  const C* __restrict__ tab = static_cast<const C*>(a.stw) + s.tw;
  C v[NB][R];
  int ob[NB];
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int b = threadIdx.x + q * blockDim.x;
    ob[q] = -1;
    if (b < total) {
      const int t = s.div_sig.div(b), low = b - t * s.sig;
      const int hi = s.div_aR.div(t), j = t - hi * s.aR;
      const int base = hi * s.blk + low;
      int k = 0;
      C w[NP];
      if (s.Ns > 1) {
        k = j - s.div_Ns.div(j) * s.Ns;
#pragma unroll
        for (int p = 0; p < NP; ++p) w[p] = __ldg(tab + p * s.Ns + k);
      }
      const int x = base + j * s.sig;
      const C* src = sm + x + s.ipad * s.div_in.div(x);
#pragma unroll
      for (int r = 0; r < R; ++r) v[q][r] = src[r * istep];
      if constexpr (kMixFused<C, R>) {
        if (s.Ns > 1)
          fused_dft<C, R>(v[q], w);
        else
          mdft<C, R>(v[q]);
      } else {
        if (s.Ns > 1) mix_twiddle<C, R>(v[q], w);
        mdft<C, R>(v[q]);
      }
      const int y = base + ((j - k) * R + k) * s.sig;
      ob[q] = y + s.opad * s.div_out.div(y);
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NB; ++q)
    if (ob[q] >= 0) {
#pragma unroll
      for (int r = 0; r < R; ++r) sm[ob[q] + r * ostep] = v[q][r];
    }
  __syncthreads();
}

// ---- a prime radix R >= 11, in the order of a primitive root g of R.  With
// x'_r the twiddled inputs, h = (R - 1) / 2 and r_m = g^m mod R, so that
// R - r_m = r_{m+h}, a pre-pass stores a_m = x'_{r_m} + x'_{R - r_m} and b_m =
// x'_{r_m} - x'_{R - r_m} at slots 1 + m and 1 + h + m of the butterfly (slot 0
// keeps x_0).  For q = r_n (n < h), r_m q = g^{m+n}; with P[t] =
// exp(-2 pi i g^t / R) = (c_t, -s_t)
//     A = x_0 + sum_m a_m c_{m+n},   B = sum_m b_m (-s_{m+n}),
//     y_q = A + i B,   y_{R-q} = A - i B,   y_0 = x_0 + sum_m a_m.
// A work item takes Q consecutive n of one butterfly: a_m and b_m are read once
// for its Q outputs and the Q roots slide by one entry per step, so a step is
// three shared-memory reads for 4 Q multiply-adds (in 2 Q packed instructions);
// the reads bound it, hence the wide items wherever every item has a thread (six
// pairs: eight spill, 2.36 against 2.33 ms for the mix below).
//
// In complex128 the two multiply-adds a clock of an SM bound it.  Items of four
// pairs pad h less; y_0 is summed by the first item of a butterfly alone, after its
// pairs (two additions beside sixteen multiply-adds in the step of every item were an
// eighth of the work); and the planner picks the threads and pencils whose warps the
// schedulers share evenly (direct_time of fft_plan.cu).  [[1021, 0], [0, 1021]] x 4, one
// direction: 17.75 ms with six pairs an item and y_0 in each, 14.58 now (0.95 of the
// multiply-add rate); a mix of 256 patterns of sides up to 512: 10.2 -> 9.4 ms.
template <typename C>
__device__ __forceinline__ void mix_locate(const MixStage& s, int b, int& base, int& j, int& k) {
  const int t = s.div_sig.div(b), low = b - t * s.sig;
  const int hi = s.div_aR.div(t);
  j = t - hi * s.aR;
  base = hi * s.blk + low;
  k = s.Ns > 1 ? j - s.div_Ns.div(j) * s.Ns : 0;
}

template <typename C, int NQ, int Q>
__device__ __noinline__ void mix_direct_pairs(C* sm, const MixStage& s, int nbf, const C* P, const int* gp) {
  using Rl = decltype(C::x);
  const int R = s.tw, h = (R - 1) / 2;
  const int istep = s.aR * s.sig, ostep = s.Ns * s.sig;
  const int items = nbf * ((h + Q - 1) / Q);
  C A[NQ][Q], B[NQ][Q], y0[NQ];
  int ob[NQ], n0[NQ];
#pragma unroll
  for (int u = 0; u < NQ; ++u) {
    const int w = threadIdx.x + u * blockDim.x;
    ob[u] = -1;
    n0[u] = 0;
    if (w < items) {
      const int blk = s.div_nb.div(w);
      int base, j, k;
      mix_locate<C>(s, w - blk * nbf, base, j, k);
      const C* pa = sm + base + j * s.sig;
      const C x0 = *pa;
      y0[u] = x0;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        A[u][i] = x0;
        B[u][i] = cmake<C>(Rl(0), Rl(0));
      }
      pa += istep;
      const C* pb = pa + h * istep;
      const C* pt = P + blk * Q;
      C wv[Q];
#pragma unroll
      for (int i = 0; i + 1 < Q; ++i) wv[i + 1] = pt[i];
      pt += Q - 1;
#pragma unroll Q
      for (int m = 0; m < h; ++m) {
#pragma unroll
        for (int i = 0; i + 1 < Q; ++i) wv[i] = wv[i + 1];
        wv[Q - 1] = *pt++;
        const C av = *pa, bv = *pb;
        pa += istep;
        pb += istep;
        if constexpr (sizeof(C) == 8) y0[u] = bsum<true>(y0[u], av);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          A[u][i] = cfma_r(av, wv[i].x, A[u][i]);
          B[u][i] = cfma_r(bv, wv[i].y, B[u][i]);
        }
      }
      if (sizeof(C) == 16 && blk == 0) {
        pa = sm + base + j * s.sig + istep;
#pragma unroll 4
        for (int m = 0; m < h; ++m, pa += istep) y0[u] = cadd(y0[u], *pa);
      }
      ob[u] = base + ((j - k) * R + k) * s.sig;
      n0[u] = blk * Q;
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < NQ; ++u) {
    if (ob[u] < 0) continue;
    if (n0[u] == 0) sm[ob[u]] = y0[u];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const int n = n0[u] + i;
      if (n < h) {
        const int q = gp[n];
        sm[ob[u] + q * ostep] = cmake<C>(A[u][i].x - B[u][i].y, A[u][i].y + B[u][i].x);
        sm[ob[u] + (R - q) * ostep] = cmake<C>(A[u][i].x + B[u][i].y, A[u][i].y - B[u][i].x);
      }
    }
  }
  __syncthreads();
}

template <typename C>
__device__ __noinline__ void mix_direct(C* sm, const MixDesc& a, const MixStage& s) {
  constexpr int NA = kMixPoints / 2;
  const int R = s.tw, h = (R - 1) / 2;
  const int nbf = a.n / R;
  const int nthr = blockDim.x;
  const int istep = s.aR * s.sig;
  const C* __restrict__ tw = static_cast<const C*>(a.tw);
  // tables after the tile: P[t], t < R - 1 + kMixWide (the sliding roots run past R - 2), then g^t mod R
  C* P = sm + a.dir_off;
  int* gp = reinterpret_cast<int*>(P + (R - 1 + kMixWide));
  const int wstride = a.tw_n / R;
  for (int e = threadIdx.x; e < R - 1 + kMixWide; e += nthr) {
    const int g = __ldg(a.gtab + s.gen + (e < R - 1 ? e : e - (R - 1)));
    P[e] = __ldg(tw + g * wstride);
    if (e < R - 1) gp[e] = g;
  }
  __syncthreads();
  {
    C av[NA], bv[NA];
    int dst[NA];
#pragma unroll
    for (int u = 0; u < NA; ++u) {
      const int w = threadIdx.x + u * nthr;
      dst[u] = -1;
      if (w < nbf * h) {
        const int m = s.div_nb.div(w);
        int base, j, k;
        mix_locate<C>(s, w - m * nbf, base, j, k);
        const int i0 = base + j * s.sig;
        const int r = gp[m];
        C x0 = sm[i0 + r * istep];
        C x1 = sm[i0 + (R - r) * istep];
        if (s.Ns > 1) {  // r k < Ns R: no reduction
          x0 = cmul(x0, __ldg(tw + (r * k) * s.twstep));
          x1 = cmul(x1, __ldg(tw + ((R - r) * k) * s.twstep));
        }
        av[u] = bsum<true>(x0, x1);
        bv[u] = bdiff<true>(x0, x1);
        dst[u] = i0 + (1 + m) * istep;
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < NA; ++u)
      if (dst[u] >= 0) {
        sm[dst[u]] = av[u];
        sm[dst[u] + h * istep] = bv[u];
      }
    __syncthreads();
  }
  constexpr int W = sizeof(C) == 8 ? kMixWide : kMixNarrow;
  if (nbf * ((h + W - 1) / W) <= nthr)
    mix_direct_pairs<C, 1, W>(sm, s, nbf, P, gp);
  else
    mix_direct_pairs<C, kMixItems, kMixNarrow>(sm, s, nbf, P, gp);
}

// The stages come sorted (direct ones first, then in the order of kMixOrder: a
// first stage of an odd radix of nine or more needs no padding; stages of one axis
// may run in any order and different axes commute), one loop per radix: a switch
// inside one loop made the compiler spill every butterfly at its barrier.  The
// radices are tested in groups of their rank, so that a pass of three stages does
// not make fifteen tests.
template <typename C, int R>
__device__ __forceinline__ void mix_stages_of(C* sm, const MixDesc& a, int& i, int& R_next) {
#pragma unroll 1
  while (R_next == R) {
    mix_stage<C, R>(sm, a, a.st[i]);
    ++i;
    R_next = i < a.nstages ? a.st[i].R : 0;
  }
}
template <typename C, int R0, int R1, int R2, int R3>
__device__ __forceinline__ void mix_stages_of4(C* sm, const MixDesc& a, int& i, int& R) {
  if (!((1 << R) & ((1 << R0) | (1 << R1) | (1 << R2) | (1 << R3)))) return;
  mix_stages_of<C, R0>(sm, a, i, R);
  mix_stages_of<C, R1>(sm, a, i, R);
  mix_stages_of<C, R2>(sm, a, i, R);
  mix_stages_of<C, R3>(sm, a, i, R);
}

template <typename C>
__device__ __forceinline__ void mix_stages(C* sm, const MixDesc& a) {
  int i = 0, R = a.nstages ? a.st[0].R : 0;
#pragma unroll 1
  while (R >= kMixMinDirect) {
    mix_direct<C>(sm, a, a.st[i]);
    ++i;
    R = i < a.nstages ? a.st[i].R : 0;
  }
  mix_stages_of4<C, 15, 13, 11, 9>(sm, a, i, R);
  mix_stages_of4<C, 16, 14, 12, 10>(sm, a, i, R);
  mix_stages_of4<C, 8, 7, 6, 5>(sm, a, i, R);
  mix_stages_of<C, 4>(sm, a, i, R);
  mix_stages_of<C, 3>(sm, a, i, R);
  mix_stages_of<C, 2>(sm, a, i, R);
}

// ---------------------------------------------------------- loads and stores
// The indices of an access cost as much as the butterflies if every element
// finds its own from tables, so the loops below step them: the box slots of a
// thread's consecutive elements differ by one fixed box point (its step times a
// generator, whatever wraps in between), the workspace is linear, and the bounds
// are clamped or predicated instead of branched on.
constexpr int kMixChunk = 4;  // global accesses of a thread in flight together

// Keeps a launch constant in a register: the compiler otherwise reloads it from
// the constant bank at every use of an unrolled loop.
__device__ __forceinline__ int pinned(int x) {
  asm("" : "+r"(x));
  return x;
}
__device__ __forceinline__ FastDiv pinned(FastDiv f) {
  asm("" : "+r"(f.mul));
  asm("" : "+r"(f.shift));
  return f;
}

template <bool COH, typename C>
__device__ __forceinline__ C mix_ld(const C* p) {
  if constexpr (COH) return __ldcg(p);
  return __ldg(p);
}

__device__ __forceinline__ float2 mix_scale(float2 v, float sx, float sy) { return __fmul2_rn(v, make_float2(sx, sy)); }
__device__ __forceinline__ double2 mix_scale(double2 v, double sx, double sy) { return make_double2(v.x * sx, v.y * sy); }

// reduce(a + b) of two box points, the point itself (the corrections of
// box_sum_slot_t).
template <int DIM>
__device__ __forceinline__ void box_sum_point(const BoxDesc& B, int* y, const int* a, const int* b) {
#pragma unroll
  for (int r = 0; r < 4; ++r) y[r] = r < DIM ? a[r] + b[r] : 0;
  if constexpr (DIM == 1) {
    y[0] -= y[0] >= B.H[0][0] ? B.H[0][0] : 0;
  } else if constexpr (DIM == 2) {
    const int c1 = y[1] >= B.H[1][1];
    y[1] -= c1 * B.H[1][1];
    y[0] -= c1 * B.H[0][1];
    y[0] += (y[0] < 0) * B.H[0][0];
    y[0] -= (y[0] >= B.H[0][0]) * B.H[0][0];
  } else if constexpr (DIM == 3) {
    const int c2 = y[2] >= B.H[2][2];
    y[2] -= c2 * B.H[2][2];
    y[1] -= c2 * B.H[1][2];
    y[0] -= c2 * B.H[0][2];
    const int c1 = (y[1] >= B.H[1][1]) - (y[1] < 0);
    y[1] -= c1 * B.H[1][1];
    y[0] -= c1 * B.H[0][1];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      y[0] += (y[0] < 0) * B.H[0][0];
      y[0] -= (y[0] >= B.H[0][0]) * B.H[0][0];
    }
  } else {
    box_fix(B, y);
  }
}

// Phase exp(-2 pi i lambda_a mu_b / n) of a split last cycle (fs_twiddle of fft_plan.hpp).
template <typename C>
__device__ __forceinline__ C mix_phase(const MixDesc& a, int la, int mu) {
  const int t = la * mu;
  return cmul(__ldg(static_cast<const C*>(a.fs_hi) + (t >> 11)), __ldg(static_cast<const C*>(a.fs_lo) + (t & 2047)));
}

// A thread's elements w0 + u nthr of a tile side of n elements.  addr(u, w)
// gives the global index of its u-th element, pos(u, w) its tile position (both
// called in order, w clamped to the tile), ok(w) whether it exists; value(v, w)
// converts.
template <typename C, bool LOAD, bool COH, typename Addr, typename Pos, typename Ok, typename Value>
__device__ __forceinline__ void mix_move(int n, const C* __restrict__ in, C* __restrict__ out, C* sm, Addr addr,
                                         Pos pos, Ok ok, Value value) {
  const int nthr = pinned(blockDim.x);
  n = pinned(n);
#pragma unroll 1
  for (int w0 = threadIdx.x; w0 < n; w0 += kMixChunk * nthr) {
    C v[kMixChunk];
    int x[kMixChunk];
#pragma unroll
    for (int u = 0; u < kMixChunk; ++u) {
      const int w = min(w0 + u * nthr, n - 1);
      if constexpr (LOAD) {
        v[u] = mix_ld<COH>(in + addr(w));
        x[u] = pos(w);
      } else {
        v[u] = sm[pos(w)];
        x[u] = addr(w);
      }
    }
#pragma unroll
    for (int u = 0; u < kMixChunk; ++u) {
      const int w = w0 + u * nthr;
      const C y = value(v[u], min(w, n - 1));
      if (w < n && ok(w)) (LOAD ? sm : out)[x[u]] = y;
    }
  }
}

// Row tiles against a box.  H side (MODE MAP_BOX_H): along the elements of one
// row, or along the rows of a [element][row] tile, by steps; otherwise each
// element from the tables.
template <typename C, int DIM, int MODE, bool LOAD>
__device__ __forceinline__ void mix_row_box(const MixDesc& a, int tile, const C* __restrict__ in,
                                            C* __restrict__ out, C* sm) {
  using Rl = decltype(C::x);
  constexpr int TS = DIM <= 2 ? 2 : 4;
  const int r0 = tile * a.T, n = a.n, nD = a.nD, T = a.T, logT = a.logT, rows = a.LB - r0;
  const Rl sx = LOAD ? Rl(1) : Rl(a.scale), sy = (LOAD ? a.conj_in : a.conj_out) ? -sx : sx;
  const int pad = pinned(a.pad);
  const FastDiv dp = pinned(a.div_pad);
  auto value = [&](C v, int) { return mix_scale(v, sx, sy); };
  auto where = [&](int x) { return LOAD ? x : x + pad * dp.div(x); };
  if (MODE == MAP_BOX_H && DIM <= 3 && (a.lay || T == 1)) {
    const int t = threadIdx.x & (T - 1), e = threadIdx.x >> logT, step = blockDim.x >> logT;
    int p[4], q[4], y[4], c[4];
    load_point<TS>(a.Atab, r0 + min(t, rows - 1), p);
    load_point<TS>(a.Btab, min(e, nD - 1), q);
    box_sum_point<DIM>(a.boxH, y, p, q);
    load_point<TS>(a.Btab, step < nD ? step : 0, c);
    BoxWalk<DIM> walk(a.boxH, y, c, a.m);
    mix_move<C, LOAD, false>(
        n, in, out, sm,
        [&](int) {
          const int s = walk.slot;
          walk.step();
          return s;
        },
        where, [&](int) { return t < rows; }, value);
    return;
  }
  const FastDiv dn = a.divnD;
  auto split = [&](int w, int& t, int& e) {
    if (MODE != MAP_WS && a.lay) {
      e = w >> logT;
      t = w - (e << logT);
    } else {
      t = dn.div(w);
      e = w - t * nD;
    }
  };
  mix_move<C, LOAD, false>(
      n, in, out, sm,
      [&](int w) {
        int t, e, p[4], q[4];
        split(w, t, e);
        const int row = r0 + min(t, rows - 1);
        load_point<TS>(MODE == MAP_BOX_H ? a.Atab : a.Ctab, row, p);
        load_point<TS>(MODE == MAP_BOX_H ? a.Btab : a.Etab, e, q);
        return box_sum_slot_t<DIM>(MODE == MAP_BOX_H ? a.boxH : a.boxG, p, q);
      },
      [&](int w) {
        if (MODE == MAP_BOX_H) return where(w);
        int t, e;
        split(w, t, e);
        const int x = __ldg(a.PIinv + e);
        return where(a.lay ? (x << logT) + t : t * nD + x);
      },
      [&](int w) {
        int t, e;
        split(w, t, e);
        return t < rows;
      },
      value);
}

// Row tiles against the workspace, where rows are contiguous; an element's tile
// position comes from the table of its column position (psin, psout).  The lanes run along a row; in a [element][row] tile of at least
// four rows, over four adjacent elements of each row in turn, which are four
// adjacent banks per row in the tile and one 32-byte sector in the workspace.
// FS: a split last cycle, whose phase is applied here.
template <typename C, bool LOAD, bool FS>
__device__ __forceinline__ void mix_row_ws(const MixDesc& a, int tile, const C* __restrict__ in, C* __restrict__ out,
                                           C* sm) {
  using Rl = decltype(C::x);
  const int r0 = tile * a.T, nD = pinned(a.nD), rows = a.LB - r0;
  const int* __restrict__ ps = LOAD ? a.psin : a.psout;
  const Rl sy = (LOAD ? a.conj_in : 0) ? Rl(-1) : Rl(1);
  if constexpr (FS) {
    // blockDim.x is a multiple of 4 T (mix_configure): a thread keeps its row
    const int logT = pinned(a.logT), quad = a.T >= 4 ? 2 : 0, sh = quad + logT, mq = (1 << quad) - 1;
    const int t = (threadIdx.x >> quad) & (a.T - 1);
    const bool live = t < rows;
    const int row = r0 + (live ? t : 0);
    const int la = row - a.fs_div.div(row) * a.fs_na, base = row * nD;
    const int n = ((nD + mq) >> quad) << sh;
    const int* __restrict__ mu = a.PIinv;
    auto elem = [&](int w) { return min(((w >> sh) << quad) | (w & mq), nD - 1); };
    mix_move<C, LOAD, false>(
        n, in, out, sm, [&](int w) { return base + elem(w); },
        [&](int w) { return (__ldg(ps + elem(w)) << logT) + t; },
        [&](int w) { return live && (((w >> sh) << quad) | (w & mq)) < nD; },
        [&](C v, int w) {
          if constexpr (LOAD) v = mix_scale(v, Rl(1), sy);
          return cmul(v, mix_phase<C>(a, la, __ldg(mu + elem(w))));
        });
  } else {
    const int pitch = LOAD ? a.pitch_in : a.pitch_out, base = r0 * nD;
    const FastDiv dn = pinned(a.divnD);
    auto value = [&](C v, int) { return LOAD ? mix_scale(v, Rl(1), sy) : v; };
    auto ok = [](int) { return true; };
    auto addr = [&](int w) { return base + w; };
    if (a.T == 1)
      mix_move<C, LOAD, false>(nD, in, out, sm, addr, [&](int w) { return __ldg(ps + w); }, ok, value);
    else
      mix_move<C, LOAD, false>(
          min(a.T, rows) * nD, in, out, sm, addr,
          [&](int w) {
            const int t = dn.div(w);
            return __ldg(ps + (w - t * nD)) + t * pitch;
          },
          ok, value);
  }
}

// Column tiles against the workspace: T adjacent columns of every row.
template <typename C, bool LOAD, bool COH>
__device__ __forceinline__ void mix_col_ws(const MixDesc& a, int tile, const C* __restrict__ in, C* __restrict__ out,
                                           C* sm) {
  using Rl = decltype(C::x);
  const int p0 = tile << a.logT, logT = pinned(a.logT), nD = pinned(a.nD), pad = pinned(a.pad);
  const FastDiv dp = pinned(a.div_pad);
  const int tcol = threadIdx.x & (a.T - 1);
  const bool live = p0 + tcol < nD;  // the last tile may hold fewer than T columns
  const int col = live ? p0 + tcol : 0;
  const Rl sy = LOAD && a.conj_in ? Rl(-1) : Rl(1);
  mix_move<C, LOAD, COH>(
      a.n, in, out, sm, [&](int w) { return (w >> logT) * nD + col; },
      [&](int w) { return LOAD ? w : w + pad * dp.div(w); }, [&](int) { return live; },
      [&](C v, int) { return LOAD ? mix_scale(v, Rl(1), sy) : v; });
}

// Column tiles against the box of G(M^T).  A thread keeps one column, and the
// columns walk the pencil sheared so that the T columns of a step are
// consecutive slots: step j of a column with axis offsets off visits row
// j + off (wrapped per axis), whose point is C[j] + (C[off] + E[column]).
template <typename C, int DIM, bool LOAD>
__device__ __forceinline__ void mix_col_box(const MixDesc& a, int tile, const C* __restrict__ in,
                                            C* __restrict__ out, C* sm) {
  using Rl = decltype(C::x);
  constexpr int TS = DIM <= 2 ? 2 : 4;
  const int p0 = tile << a.logT, logT = pinned(a.logT), pad = pinned(a.pad), nsub = a.nsub, LB = pinned(a.LB);
  const FastDiv dp = pinned(a.div_pad);
  const int tcol = threadIdx.x & (a.T - 1);
  const bool live = p0 + tcol < a.nD;
  const Rl sx = LOAD ? Rl(1) : Rl(a.scale), sy = (LOAD ? a.conj_in : a.conj_out) ? -sx : sx;
  int off[kMaxSub] = {0, 0, 0}, row = 0;
#pragma unroll
  for (int s = 0; s < kMaxSub; ++s)
    if (s < nsub) {
      off[s] = a.sub_div[s].mod(tcol * a.alpha[s]);
      row = row * a.sub_n[s] + off[s];
    }
  int f[4], p[4], q[4];
  load_point<TS>(a.Ctab, row, p);
  load_point<TS>(a.Etab, live ? p0 + tcol : 0, q);
  box_sum_point<DIM>(a.boxG, f, p, q);
  auto value = [&](C v, int) { return mix_scale(v, sx, sy); };
  auto ok = [&](int) { return live; };
  auto where = [&](int i) {
    const int x = (i << logT) + tcol;
    return LOAD ? x : x + pad * dp.div(x);
  };
  if (DIM <= 3 && nsub == 1) {
    const int j0 = threadIdx.x >> logT, step = blockDim.x >> logT;
    int y[4], c[4];
    load_point<TS>(a.Ctab, min(j0, LB - 1), p);
    box_sum_point<DIM>(a.boxG, y, p, f);
    load_point<TS>(a.Ctab, step < LB ? step : 0, c);
    BoxWalk<DIM> walk(a.boxG, y, c, a.m);
    mix_move<C, LOAD, false>(
        a.n, in, out, sm,
        [&](int) {
          const int s = walk.slot;
          walk.step();
          return s;
        },
        [&](int w) {
          const int i = (w >> logT) + off[0];
          return where(i >= LB ? i - LB : i);
        },
        ok, value);
    return;
  }
  const int n1 = pinned(a.sub_n[nsub - 1]), o1 = nsub == 1 ? off[0] : nsub == 2 ? off[1] : off[2];
  const int n0 = a.sub_n[nsub >= 2 ? nsub - 2 : 0], o0 = nsub == 2 ? off[0] : off[1];
  const FastDiv d1 = pinned(a.sub_div[nsub - 1]), d0 = a.sub_div[nsub >= 2 ? nsub - 2 : 0];
  mix_move<C, LOAD, false>(
      a.n, in, out, sm,
      [&](int w) {
        int ct[4];
        load_point<TS>(a.Ctab, w >> logT, ct);
        return box_sum_slot_t<DIM>(a.boxG, ct, f);
      },
      [&](int w) {
        const int j = w >> logT;
        int r = d1.div(j);
        int i1 = j - r * n1 + o1;
        if (i1 >= n1) i1 -= n1;
        if (nsub == 1) return where(i1);
        int i0 = r;
        if (nsub == 3) {
          r = d0.div(i0);
          i0 -= r * n0;
        }
        i0 += o0;
        if (i0 >= n0) i0 -= n0;
        if (nsub == 3) {
          int i2 = r + off[0];
          if (i2 >= a.sub_n[0]) i2 -= a.sub_n[0];
          i0 += i2 * n0;
        }
        return where(i0 * n1 + i1);
      },
      ok, value);
}

// Whole tiles: T consecutive signals in slot order.
template <typename C, bool LOAD>
__device__ __forceinline__ void mix_whole_io(const MixDesc& a, int tile, const C* __restrict__ in,
                                             C* __restrict__ out, C* sm) {
  using Rl = decltype(C::x);
  const int* __restrict__ map = (LOAD ? a.load_mode : a.store_mode) == MAP_BOX_H ? a.map_in : a.map_out;
  const int b0 = tile * a.T, L = pinned(a.L), pad = pinned(a.pad);
  const FastDiv dL = pinned(a.divL), dp = pinned(a.div_pad);
  const Rl sx = LOAD ? Rl(1) : Rl(a.scale), sy = (LOAD ? a.conj_in : a.conj_out) ? -sx : sx;
  const int64_t base = (int64_t)b0 * L;
  mix_move<C, LOAD, false>(
      min(a.T, a.batch - b0) * L, in + base, out + base, sm, [](int w) { return w; },
      [&](int w) {
        const int t = dL.div(w);
        const int x = t * L + __ldg(map + (w - t * L));
        return LOAD ? x : x + pad * dp.div(x);
      },
      [](int) { return true; }, [&](C v, int) { return mix_scale(v, sx, sy); });
}

template <typename C, int DIM, bool LOAD>
__device__ __forceinline__ void mix_io_box(const MixDesc& a, int tile, const C* __restrict__ in, C* __restrict__ out,
                                           C* sm) {
  if (a.kind == MIX_COL)
    mix_col_box<C, DIM, LOAD>(a, tile, in, out, sm);
  else if ((LOAD ? a.load_mode : a.store_mode) == MAP_BOX_H)
    mix_row_box<C, DIM, MAP_BOX_H, LOAD>(a, tile, in, out, sm);
  else
    mix_row_box<C, DIM, MAP_BOX_G, LOAD>(a, tile, in, out, sm);
}

template <typename C, bool LOAD, bool COH>
__device__ __forceinline__ void mix_io(const MixDesc& a, int tile, const C* __restrict__ in, C* __restrict__ out,
                                       C* sm) {
  if (a.kind == MIX_WHOLE) return mix_whole_io<C, LOAD>(a, tile, in, out, sm);
  if ((LOAD ? a.load_mode : a.store_mode) == MAP_WS) {
    if (a.kind == MIX_COL) return mix_col_ws<C, LOAD, COH>(a, tile, in, out, sm);
    if (a.lay) return mix_row_ws<C, LOAD, true>(a, tile, in, out, sm);
    return mix_row_ws<C, LOAD, false>(a, tile, in, out, sm);
  }
  switch (a.d) {
    case 1: return mix_io_box<C, 1, LOAD>(a, tile, in, out, sm);
    case 2: return mix_io_box<C, 2, LOAD>(a, tile, in, out, sm);
    case 3: return mix_io_box<C, 3, LOAD>(a, tile, in, out, sm);
    default: return mix_io_box<C, 4, LOAD>(a, tile, in, out, sm);
  }
}

// One tile of signal sig.  COH: the workspace was written by other CTAs of
// the same launch (read through the L2).
template <typename C, bool COH>
__device__ __forceinline__ void mixed_body(const MixDesc& a, int tile, int sig, C* sm) {
  const C* in = static_cast<const C*>(a.in) + (int64_t)sig * a.m;
  C* out = static_cast<C*>(a.out) + (int64_t)sig * a.m;
  mix_io<C, true, COH>(a, tile, in, out, sm);
  __syncthreads();
  mix_stages<C>(sm, a);
  mix_io<C, false, false>(a, tile, in, out, sm);
}

template <typename C>
__global__ void __launch_bounds__(kMixThreads<C>, 1) mixed_kernel(const __grid_constant__ MixDesc a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  mixed_body<C, false>(a, blockIdx.x, blockIdx.y, reinterpret_cast<C*>(smem_raw));
}

}  // namespace pfft
