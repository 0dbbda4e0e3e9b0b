// fft.cuh -- block-wide power-of-two complex FFTs in shared memory.
//
// Stockham autosort formulation (natural-order input and output, no bit
// reversal): pass p with stride Ns = R_0 R_1 ... R_{p-1} and radix R maps,
// for every j in [0, N/R) with k = j mod Ns,
//   v_r = x[j + r N/R] * w^{r k},  w = exp(sigma 2 pi i / (Ns R)),
//   y[(j - k) R + k + q Ns] = sum_r v_r exp(sigma 2 pi i r q / R).
// Radix-8 passes first, then one radix-4 or radix-2 pass for the remaining
// bits.  Each thread owns exactly 8 elements per pass (one radix-8 butterfly,
// two radix-4 or four radix-2 butterflies), so a block of B transforms of
// length N runs with B*N/8 threads.  The pass reads all of its elements into
// registers, synchronises, then writes in place.
//
// Transform b lives at buf + b*bstride, element n at sidx<T>(n).  Twiddles come
// from a pass-ordered table: the pass with stride Ns and radix R reads
//   tw[r*Ns + k - 1] = exp(-2 pi i r k / (Ns R)),  1 <= r < R, 0 <= k < Ns,
// (rows r of Ns consecutive entries; the index ranges of successive passes
// tile [0, N-1)), so a warp's loads for one r are contiguous.  The table is
// computed in FP64 on the host (fft_twiddle_table) and rounded to T; the
// inverse transform (sigma = +1) uses its conjugate.  No normalisation.
// The FP64 group transforms (gfft) run in 64-bit block fixed point
// (fft64.cuh) with a table of their own in the same order.
#pragma once
#include <cmath>
#include <vector>

#include "common.cuh"
#include "fft64.cuh"

namespace lm {

template <typename T, int SIGN>
__device__ __forceinline__ cplx<T> mul_sigma_i(cplx<T> a) {  // a * (sigma i)
  return SIGN > 0 ? mk<T>(-a.y, a.x) : mk<T>(a.y, -a.x);
}

template <typename T, int SIGN>
__device__ __forceinline__ void dft4(cplx<T>& a0, cplx<T>& a1, cplx<T>& a2, cplx<T>& a3) {
  cplx<T> t0 = cadd<T>(a0, a2), t1 = csub<T>(a0, a2);
  cplx<T> t2 = cadd<T>(a1, a3), t3 = mul_sigma_i<T, SIGN>(csub<T>(a1, a3));
  a0 = cadd<T>(t0, t2);
  a2 = csub<T>(t0, t2);
  a1 = cadd<T>(t1, t3);
  a3 = csub<T>(t1, t3);
}

template <typename T, int SIGN>
__device__ __forceinline__ void dft8(cplx<T>* v) {
  cplx<T> a0 = v[0], a1 = v[2], a2 = v[4], a3 = v[6];
  cplx<T> b0 = v[1], b1 = v[3], b2 = v[5], b3 = v[7];
  dft4<T, SIGN>(a0, a1, a2, a3);
  dft4<T, SIGN>(b0, b1, b2, b3);
  const T h = (T)0.70710678118654752440;
  // b_q *= exp(sigma 2 pi i q / 8)
  b1 = mk<T>((b1.x - SIGN * b1.y) * h, (SIGN * b1.x + b1.y) * h);
  b2 = mul_sigma_i<T, SIGN>(b2);
  b3 = mk<T>((-b3.x - SIGN * b3.y) * h, (SIGN * b3.x - b3.y) * h);
  v[0] = cadd<T>(a0, b0); v[4] = csub<T>(a0, b0);
  v[1] = cadd<T>(a1, b1); v[5] = csub<T>(a1, b1);
  v[2] = cadd<T>(a2, b2); v[6] = csub<T>(a2, b2);
  v[3] = cadd<T>(a3, b3); v[7] = csub<T>(a3, b3);
}

// Twiddles w^{r k}, 1 <= r < R, w = exp(sigma 2 pi i / (Ns R)), of one
// butterfly, all from the table (FP64 multiplies are the scarce resource).
template <typename T, int SIGN, int R>
__device__ __forceinline__ void butterfly_twiddles(cplx<T>* w, int k, int lNs, const cplx<T>* __restrict__ tw) {
  const cplx<T>* t = tw + (k - 1);
#pragma unroll
  for (int r = 1; r < R; ++r) {
    w[r] = __ldg(t + (r << lNs));
    if (SIGN > 0) w[r].y = -w[r].y;
  }
}

template <typename T, int SIGN, int LR>
__device__ __forceinline__ void stockham_pass(cplx<T>* buf, int log2N, int lNs, int bstride,
                                              const cplx<T>* __restrict__ tw) {
  constexpr int R = 1 << LR;
  constexpr int NB = 8 / R;  // butterflies per thread
  const int lNR = log2N - LR;
  const int NR = 1 << lNR;
  const int Ns = 1 << lNs;
  const int nthr = blockDim.x;
  cplx<T> v[8];
  int base[NB], outb[NB];
#pragma unroll
  for (int u = 0; u < NB; ++u) {
    const int g = u * nthr + threadIdx.x;
    const int b = g >> lNR;
    const int j = g & (NR - 1);
    const int k = j & (Ns - 1);
    const cplx<T>* src = buf + b * bstride;
    base[u] = b * bstride;
    outb[u] = ((j - k) << LR) + k;
#pragma unroll
    for (int r = 0; r < R; ++r) v[u * R + r] = src[sidx<T>(j + r * NR)];
    if (k > 0) {
      cplx<T> w[R];
      butterfly_twiddles<T, SIGN, R>(w, k, lNs, tw);
#pragma unroll
      for (int r = 1; r < R; ++r) v[u * R + r] = cmul<T>(v[u * R + r], w[r]);
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < NB; ++u) {
    cplx<T>* vv = v + u * R;
    if (LR == 3) {
      dft8<T, SIGN>(vv);
    } else if (LR == 2) {
      dft4<T, SIGN>(vv[0], vv[1], vv[2], vv[3]);
    } else {
      cplx<T> a = vv[0], b = vv[1];
      vv[0] = cadd<T>(a, b);
      vv[1] = csub<T>(a, b);
    }
#pragma unroll
    for (int q = 0; q < R; ++q) buf[base[u] + sidx<T>(outb[u] + q * Ns)] = vv[q];
  }
  __syncthreads();
}

// Block-wide FFT of `batch` transforms of length 2^log2N; requires
// blockDim.x * 8 == batch * 2^log2N and log2N >= 1.  Callers synchronise
// before (data in place); the function ends with a barrier.  (FP64, for
// csrc/project_static.cu; the other transforms are group transforms.)
template <typename T, int SIGN>
__device__ void block_fft(cplx<T>* buf, int log2N, int bstride, const cplx<T>* __restrict__ tw) {
  int lNs = 0;
  int rem = log2N;
  while (rem >= 3) {
    stockham_pass<T, SIGN, 3>(buf, log2N, lNs, bstride, tw);
    lNs += 3;
    rem -= 3;
  }
  if (rem == 2) stockham_pass<T, SIGN, 2>(buf, log2N, lNs, bstride, tw);
  if (rem == 1) stockham_pass<T, SIGN, 1>(buf, log2N, lNs, bstride, tw);
}

template <typename T, int SIGN, int R>
__device__ __forceinline__ void dft_r(cplx<T>* v) {
  if (R == 8) {
    dft8<T, SIGN>(v);
  } else if (R == 4) {
    dft4<T, SIGN>(v[0], v[1], v[2], v[3]);
  } else {
    const cplx<T> a = v[0], b = v[1];
    v[0] = cadd<T>(a, b);
    v[1] = csub<T>(a, b);
  }
}

// ---------------------------------------------------------------------------
// Register-resident transforms owned by a group of G = N/8 threads (one
// transform per group; groups never wait for one another), N = 2^L fixed at
// compile time.  Thread j of the group holds elements j + m G, m < 8, of its
// transform in x[m] on entry (input) and on exit (output): the first pass's
// butterflies read exactly these positions, and the last pass's butterflies
// write them.  The passes in between exchange through two shared buffers
// used alternately, so each pass costs one group barrier.  Every stride,
// shared-memory offset and twiddle-table offset is a compile-time constant
// (with run-time lengths the index arithmetic cost more instructions than
// the butterflies), and twiddles are applied without a branch at k = 0 (the
// table holds w^0 = 1 there; the product is exact).
// SYNC: 0 the warp (G <= 32: several groups per warp execute the same
// instructions), 1 named barrier grp + 1 over the group's G threads, 2 the
// block (groups whose threads interleave, column tiles), 3 and 4 half or
// quarter grp of the block (the same, two or four sets of them).  A named barrier
// with a run-time id reserves all 16 of a block's barriers, which limits the
// blocks resident on an SM, so kernels whose groups all fit in a warp are
// compiled without it.

template <int SYNC, int G>
__device__ __forceinline__ void gsync(int grp) {
  if constexpr (SYNC == 2) __syncthreads();
  else if constexpr (SYNC >= 3) {
    const unsigned n = blockDim.x >> (SYNC - 2);
    if (grp == 0) asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory");
    else if (SYNC == 3 || grp == 1) asm volatile("bar.sync 2, %0;" ::"r"(n) : "memory");
    else if (grp == 2) asm volatile("bar.sync 3, %0;" ::"r"(n) : "memory");
    else asm volatile("bar.sync 4, %0;" ::"r"(n) : "memory");
  } else if constexpr (SYNC == 1) asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(G) : "memory");
  else __syncwarp();
}

// Twiddles w^{r k}, 1 <= r < R, of a butterfly of the pass with stride
// Ns = 2^LNS: the table's for r = 1, 2, 4, the others as products (at most two
// multiplications deep).  (At 1024^2-2048^2 the column passes ran 10-15% faster
// with the table than with sincospif.)
template <int SIGN, int R, int LNS>
__device__ __forceinline__ void twiddles_ct(float2* w, int k, const float2* __restrict__ tw) {
  const float2* t = tw + (k - 1);
  auto ev = [&](int r) {
    float2 c = __ldg(t + (r << LNS));
    if (SIGN > 0) c.y = -c.y;
    return c;
  };
  w[1] = ev(1);
  if (R >= 4) {
    w[2] = ev(2);
    w[3] = cmul<float>(w[1], w[2]);
  }
  if (R == 8) {
    w[4] = ev(4);
    w[5] = cmul<float>(w[4], w[1]);
    w[6] = cmul<float>(w[4], w[2]);
    w[7] = cmul<float>(w[4], w[3]);
  }
}

// Arithmetic of the group transforms.  FP32: float2 values.  FP64: 64-bit
// block fixed point (fft64.cuh), where pass P shifts its inputs right by sh.
struct PassShift {
  int sh, half;
};
template <int SIGN, int R, int LNS>
__device__ __forceinline__ void twiddle_ct(float2* v, int k, const float2* __restrict__ tw, PassShift) {
  float2 wr[8];
  twiddles_ct<SIGN, R, LNS>(wr, k, tw);
#pragma unroll
  for (int r = 1; r < R; ++r) v[r] = cmul<float>(v[r], wr[r]);
}
template <int SIGN, int R, int LNS>
__device__ __forceinline__ void twiddle_ct(cfx* v, int k, const TwFx* __restrict__ tw, PassShift s) {
  const int4* t = reinterpret_cast<const int4*>(tw + (k - 1));
  v[0] = fx_shift(v[0], s.sh, s.half);
#pragma unroll
  for (int r = 1; r < R; ++r) {
    const int4 q = __ldg(t + (r << LNS));
    v[r] = fx_twiddle<SIGN>(v[r], TwFx{q.x, q.y, q.z, q.w}, s.sh, s.half);
  }
}
template <int SIGN, int R> __device__ __forceinline__ void butterfly(float2* v) { dft_r<float, SIGN, R>(v); }
template <int SIGN, int R> __device__ __forceinline__ void butterfly(cfx* v) { fdft_r<SIGN, R>(v); }

// Middle pass P (radix 8, stride Ns = 8^P) from `in` to `out`.
template <typename V, typename W, int SIGN, int L, int P>
__device__ __forceinline__ void gpass8(const V* in, V* out, int j, const W* __restrict__ tw, PassShift s) {
  constexpr int G = 1 << (L - 3), LNS = 3 * P, NS = 1 << LNS;
  constexpr int RS = G + G / 8;    // shared-memory distance of G positions (G % 8 == 0)
  constexpr int WS = NS + NS / 8;  // of Ns positions
  V v[8];
  const int rb = j + (j >> 3);
#pragma unroll
  for (int r = 0; r < 8; ++r) v[r] = in[rb + r * RS];
  const int k = j & (NS - 1);
  twiddle_ct<SIGN, 8, LNS>(v, k, tw, s);
  butterfly<SIGN, 8>(v);
  const int o = ((j - k) << 3) + k;
  const int ob = o + (o >> 3);
#pragma unroll
  for (int q = 0; q < 8; ++q) out[ob + q * WS] = v[q];
}

// Last pass (radix 8, 4 or 2) from `in` into the registers x.
template <typename V, typename W, int SIGN, int L>
__device__ __forceinline__ void gpass_last(V (&x)[8], const V* in, int j, const W* __restrict__ tw, PassShift s) {
  constexpr int G = 1 << (L - 3), NP = (L + 2) / 3, P = NP - 1;
  constexpr int LNS = 3 * P, NS = 1 << LNS, LR = L - LNS, R = 1 << LR, NB = 8 / R;
  constexpr int RS = (G * NB) + (G * NB) / 8;  // distance of N/R positions (a multiple of 8)
  V v[8];
#pragma unroll
  for (int u = 0; u < NB; ++u) {
    const int jj = u * G + j;
    const int k = jj & (NS - 1);
    const int rb = jj + (jj >> 3);
#pragma unroll
    for (int r = 0; r < R; ++r) v[u * R + r] = in[rb + r * RS];
    twiddle_ct<SIGN, R, LNS>(v + u * R, k, tw, s);
  }
#pragma unroll
  for (int u = 0; u < NB; ++u) {
    butterfly<SIGN, R>(v + u * R);
#pragma unroll
    for (int q = 0; q < R; ++q) x[u + q * NB] = v[u * R + q];
  }
}

// Shift of pass P (P >= 1) when the sum bound allows Dn bits in all, and the
// bits dropped by the passes up to P.
template <int P> __device__ __forceinline__ int pass_drop(int Dn) { return Dn < 3 * P ? Dn : 3 * P; }
template <int P> __device__ __forceinline__ PassShift pass_shift(int Dn) {
  const int sh = pass_drop<P>(Dn) - pass_drop<P - 1>(Dn);
  return PassShift{sh, (1 << sh) >> 1};
}

template <typename V, typename W, int SIGN, int L, int P, int SYNC>
__device__ __forceinline__ void gpass_mid(V* buf0, V* buf1, int& w, int j, int grp, const W* __restrict__ tw,
                                          int Dn) {
  constexpr int NP = (L + 2) / 3;
  if constexpr (P < NP - 1) {
    gpass8<V, W, SIGN, L, P>(w ? buf1 : buf0, w ? buf0 : buf1, j, tw, pass_shift<P>(Dn));
    gsync<SYNC, (1 << (L - 3))>(grp);
    w ^= 1;
    gpass_mid<V, W, SIGN, L, P + 1, SYNC>(buf0, buf1, w, j, grp, tw, Dn);
  }
}

// First pass (radix 8, no twiddles) of x into the free exchange buffer.
template <typename V, int SIGN> __device__ __forceinline__ void gpass_first(V (&x)[8], V* out, int j) {
  butterfly<SIGN, 8>(x);
  const int b = 9 * j;  // sidx(8 j + q) = 9 j + q
#pragma unroll
  for (int q = 0; q < 8; ++q) out[b + q] = x[q];
}

// Reduction scratch of a block's transforms (FP64 only): the groups' warps
// leave their maxima in the first half and their sums in the second.  For
// column tiles (SYNC 2 to 4) lC: log2 of the interleaved columns, tid and n:
// the thread's index in and the threads of its set of transforms.
constexpr int GRED_WORDS = 512;
struct GRed {
  unsigned* red;
  int lC, tid, n;
};
template <typename T> struct GRedWords { static constexpr int value = sizeof(T) == 8 ? GRED_WORDS : 1; };

// Reduce v over a transform's threads: MAX or sum.  Within a warp by
// shuffles; the warps' results go to `slots`, to be combined by gred_read
// after a barrier of the group.
template <bool MAX, int SYNC, int G>
__device__ __forceinline__ unsigned gred_warp(unsigned v, unsigned* slots, int grp, const GRed& g) {
  const int lC = g.lC;
  const int lo = SYNC >= 2 ? 1 << lC : 1;
  const int hi = SYNC == 0 && G < 32 ? G / 2 : 16;
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    if (off <= hi && off >= lo) {
      const unsigned o = __shfl_xor_sync(0xffffffffu, v, off);
      v = MAX ? max(v, o) : v + o;
    }
  }
  if (SYNC == 1) {
    if ((threadIdx.x & 31) == 0) slots[grp * 16 + ((threadIdx.x % G) >> 5)] = v;
  } else if (SYNC >= 2) {
    if ((g.tid & 31) < (1 << lC)) slots[((g.tid >> 5) << lC) + (g.tid & 31)] = v;
  }
  return v;
}
template <bool MAX, int SYNC, int G>
__device__ __forceinline__ unsigned gred_read(unsigned v, const unsigned* slots, int grp, const GRed& g) {
  if (SYNC == 1) {
    v = 0;
#pragma unroll
    for (int i = 0; i < G / 32; ++i) v = MAX ? max(v, slots[grp * 16 + i]) : v + slots[grp * 16 + i];
  } else if (SYNC >= 2) {
    const int nw = g.n >> 5, c = g.tid & ((1 << g.lC) - 1);
    v = 0;
    for (int i = 0; i < nw; ++i) v = MAX ? max(v, slots[(i << g.lC) + c]) : v + slots[(i << g.lC) + c];
  }
  return v;
}

// The transform of x (positions j + m G in, positions j + m G out), times
// 2^sc; w selects the exchange buffer that is free to write and is left
// pointing at the buffer not read last.
template <typename T, int SIGN, int L, int SYNC>
__device__ __forceinline__ void gfft(cplx<T> (&x)[8], cplx<T>* buf0, cplx<T>* buf1, int& w, int j, int grp,
                                     const twid<T>* __restrict__ tw, GRed gr, int sc = 0) {
  static_assert(L >= 4 && L <= 11, "transform length 16..2048");
  constexpr int G = 1 << (L - 3), NP = (L + 2) / 3;
  if constexpr (sizeof(T) == 4) {
    gpass_first<float2, SIGN>(x, w ? buf1 : buf0, j);
    gsync<SYNC, G>(grp);
    gpass_mid<float2, float2, SIGN, L, 1, SYNC>(buf0, buf1, w, j, grp, tw, 0);
    gpass_last<float2, float2, SIGN, L>(x, w ? buf1 : buf0, j, tw, PassShift{0, 0});
    if (sc != 0) {
      const float f = __int_as_float((127 + sc) << 23);
#pragma unroll
      for (int m = 0; m < 8; ++m) x[m] = cscale<float>(x[m], f);
    }
  } else {
    cfx* b0 = reinterpret_cast<cfx*>(buf0);
    cfx* b1 = reinterpret_cast<cfx*>(buf1);
    unsigned mx = 0;
#pragma unroll
    for (int m = 0; m < 8; ++m) mx = max(mx, max(fx_abs_hi(x[m].x), fx_abs_hi(x[m].y)));
    mx = gred_warp<true, SYNC, G>(mx, gr.red, grp, gr);
    if (SYNC != 0) gsync<SYNC, G>(grp);
    mx = gred_read<true, SYNC, G>(mx, gr.red, grp, gr);
    const int emax = max((int)(mx >> 20), FX_EMIN);
    cfx v[8];
    unsigned ms = 0;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      v[m].x = fx_from_double(x[m].x, emax, ms);
      v[m].y = fx_from_double(x[m].y, emax, ms);
    }
    unsigned sum = gred_warp<false, SYNC, G>(fx_sum_units(ms), gr.red + GRED_WORDS / 2, grp, gr);
    gpass_first<cfx, SIGN>(v, w ? b1 : b0, j);
    gsync<SYNC, G>(grp);
    sum = gred_read<false, SYNC, G>(sum, gr.red + GRED_WORDS / 2, grp, gr);
    const int Dn = fx_sum_shift(sum);
    gpass_mid<cfx, TwFx, SIGN, L, 1, SYNC>(b0, b1, w, j, grp, tw, Dn);
    gpass_last<cfx, TwFx, SIGN, L>(v, w ? b1 : b0, j, tw, pass_shift<NP - 1>(Dn));
    // exponents near the top of the range: 2^512 below, then a product that
    // overflows as FP64 does (NaN for a transform with non-finite inputs)
    const bool top = emax > 1980;
    const int e = emax + pass_drop<NP - 1>(Dn) + sc - (top ? 512 : 0);
#pragma unroll
    for (int m = 0; m < 8; ++m) x[m] = mk<double>(fx_to_double(v[m].x, e), fx_to_double(v[m].y, e));
    if (top) {
      const double f = emax >= 2047 ? __longlong_as_double(0x7ff8000000000000LL) : 1.3407807929942597e154;
#pragma unroll
      for (int m = 0; m < 8; ++m) x[m] = cscale<double>(x[m], f);
    }
  }
  w ^= 1;
}

// Host: the pass-ordered twiddle table of an N-point transform (N - 1
// entries, FP64).
inline void fft_twiddle_table(int log2N, double* re, double* im) {
  const double twopi = 6.283185307179586476925286766559;
  int lNs = 0;
  for (int p = 0; p < fft_num_passes(log2N); ++p) {
    const int lr = fft_pass_lr(log2N, p);
    const int Ns = 1 << lNs, R = 1 << lr;
    for (int r = 1; r < R; ++r)
      for (int k = 0; k < Ns; ++k) {
        const double a = twopi * (double)(r * k) / (double)(Ns * R);
        re[r * Ns + k - 1] = std::cos(a);
        im[r * Ns + k - 1] = -std::sin(a);
      }
    lNs += lr;
  }
}

}  // namespace lm
