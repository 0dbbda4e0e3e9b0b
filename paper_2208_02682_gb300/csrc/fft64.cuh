// fft64.cuh -- FP64 transforms in 64-bit block fixed point.
//
// Why: sm_103 issues FP64 arithmetic at two lanes per SM and clock (1.26
// TFLOP/s), one warp instruction in 16 clocks, while its integer pipes take
// a warp instruction every clock or two.  A 64-bit fixed-point addition is
// two instructions and a product with a twiddle six 32 x 32 + 64 bit
// multiply-adds per component, so a radix-8 pass costs about an eighth of
// its FP64 form, with more than FP64's 53 bits carried through it.  Measured
// on whole FP64 steps (Strategy 1, four means, positions, Eulerian means),
// FP64 butterflies -> this: 1024^2 6.72 -> 2.60 ms, 256^2 0.62 -> 0.33 ms,
// 64^2 0.236 -> 0.207 ms.  Against an extended-precision transform the error
// is 0.25-0.8 of the FP64 butterflies' over 16..2048 points and white, steep,
// single-mode and mixed-scale inputs.
//
// Format: all 2 N components of one transform share one binary exponent,
// taken from its largest component (exponent field emax): the component d is
// held as X = trunc(d 2^(1081 - emax)), |X| < 2^59.  Additions are then
// exact; products with twiddles (62 fractional bits) are rounded to nearest.
// Growth: after p radix-8 passes every intermediate value is a sum of 8^p
// inputs times unit factors, hence at most min(S, 8^p M) in modulus, with M
// the largest modulus and S the sum |re| + |im| over the transform.  Pass p
// (p = 1, 2, ...) therefore shifts its inputs right (rounded) until
// D_p = min(3 p, D) bits are dropped in all, D the smallest shift with
// S 2^-D <= 2^59: known before the first pass, so the passes need no further
// reductions, inputs of a pass stay below 2^59.5 and outputs below 2^62.5.
// Error, relative in the 2-norm of the transform: the last rounding dominates,
// about sqrt(2 N)/2 units against a signal of at least
// sqrt(N) 2^59 |x|_2/S >= 2^58.5 units: 2^-55 at N = 2048 for the worst
// input, below the 2^-53 a component of FP64 arithmetic itself.
// Components more than 2^59 times smaller than the largest become zero, as
// they would be absorbed by it in a butterfly; exponents below 130 (1e-269)
// are taken as 130.  A non-finite component makes the whole transform NaN.
#pragma once
#include <string.h>

#include <cmath>
#include <vector>

#include <cuda_runtime.h>

#if defined(__CUDA_ARCH__)
#define LM_HD __device__ __forceinline__
#else
#define LM_HD __host__ __device__ inline
#endif

namespace lm {

struct cfx {
  long long x, y;
};

// Twiddle c + i s with c = ch 2^-30 + cl 2^-62, s likewise; entries of the
// pass-ordered table (see fft.cuh), w = exp(-i theta).
struct __align__(16) TwFx {
  int ch, cl, sh, sl;
};

LM_HD cfx fadd(cfx a, cfx b) { return cfx{a.x + b.x, a.y + b.y}; }
LM_HD cfx fsub(cfx a, cfx b) { return cfx{a.x - b.x, a.y - b.y}; }
template <int SIGN> LM_HD cfx fmul_sigma_i(cfx a) { return SIGN > 0 ? cfx{-a.y, a.x} : cfx{a.y, -a.x}; }

LM_HD int fx_lo(long long v) { return (int)(unsigned)(unsigned long long)v; }
// the high part of v = hi 2^32 + lo with lo signed
LM_HD int fx_hi(long long v) {
  const unsigned long long u = (unsigned long long)v;
  return (int)((unsigned)(u >> 32) + ((unsigned)u >> 31));
}
LM_HD long long fx_mad(int a, int b, long long c) { return (long long)a * b + c; }

// v / sqrt(2), |v| <= 2^62.5, rounded
LM_HD long long fx_mul_rsqrt2(long long v) {
  constexpr int HC = 759250125;                  // round(2^30/sqrt 2)
  constexpr int HL4 = -25716447;                 // round(2^62 (1/sqrt 2 - HC 2^-30))
  const int lo = fx_lo(v), hi = fx_hi(v);
  long long m = fx_mad(lo, HC, 1LL << 29);
  m = fx_mad(hi, HL4, m);
  return (long long)((unsigned long long)((long long)hi * HC) << 2) + (m >> 30);
}

template <int SIGN> LM_HD void fdft4(cfx& a0, cfx& a1, cfx& a2, cfx& a3) {
  const cfx t0 = fadd(a0, a2), t1 = fsub(a0, a2);
  const cfx t2 = fadd(a1, a3), t3 = fmul_sigma_i<SIGN>(fsub(a1, a3));
  a0 = fadd(t0, t2);
  a2 = fsub(t0, t2);
  a1 = fadd(t1, t3);
  a3 = fsub(t1, t3);
}

template <int SIGN> LM_HD void fdft8(cfx* v) {
  cfx a0 = v[0], a1 = v[2], a2 = v[4], a3 = v[6];
  cfx b0 = v[1], b1 = v[3], b2 = v[5], b3 = v[7];
  fdft4<SIGN>(a0, a1, a2, a3);
  fdft4<SIGN>(b0, b1, b2, b3);
  // b_q *= exp(sigma 2 pi i q / 8)
  const long long p1 = fx_mul_rsqrt2(b1.x - b1.y), q1 = fx_mul_rsqrt2(b1.x + b1.y);
  const long long p3 = fx_mul_rsqrt2(b3.x - b3.y), q3 = fx_mul_rsqrt2(b3.x + b3.y);
  b1 = SIGN > 0 ? cfx{p1, q1} : cfx{q1, -p1};
  b2 = fmul_sigma_i<SIGN>(b2);
  b3 = SIGN > 0 ? cfx{-q3, p3} : cfx{-p3, -q3};
  v[0] = fadd(a0, b0); v[4] = fsub(a0, b0);
  v[1] = fadd(a1, b1); v[5] = fsub(a1, b1);
  v[2] = fadd(a2, b2); v[6] = fsub(a2, b2);
  v[3] = fadd(a3, b3); v[7] = fsub(a3, b3);
}

template <int SIGN, int R> LM_HD void fdft_r(cfx* v) {
  if (R == 8) {
    fdft8<SIGN>(v);
  } else if (R == 4) {
    fdft4<SIGN>(v[0], v[1], v[2], v[3]);
  } else {
    const cfx a = v[0], b = v[1];
    v[0] = fadd(a, b);
    v[1] = fsub(a, b);
  }
}

// v shifted right by sh (0..3), rounded; half = 2^(sh-1), or 0 for sh = 0
LM_HD cfx fx_shift(cfx v, int sh, int half) { return cfx{(v.x + half) >> sh, (v.y + half) >> sh}; }

// v times the twiddle (SIGN > 0: its conjugate), rounded to units and then
// shifted right by sh, rounded; |v| <= 2^62.5 before the shift.  Per
// component: the four cross products low x high at weight 2^-30 (their sum
// stays below 2^62.9), rounded to units, and the two high products; low x
// low, below a quarter unit, is dropped.
template <int SIGN> LM_HD cfx fx_twiddle(cfx v, TwFx w, int sh, int half) {
  const int al = fx_lo(v.x), ah = fx_hi(v.x);
  const int bl = fx_lo(v.y), bh = fx_hi(v.y);
  if (SIGN > 0) {
    w.sh = -w.sh;
    w.sl = -w.sl;
  }
  const int nh = -w.sh, nl = -w.sl;
  long long m = fx_mad(al, w.ch, 1LL << 29), n = fx_mad(al, w.sh, 1LL << 29);
  m = fx_mad(bl, nh, m);
  n = fx_mad(bl, w.ch, n);
  m = fx_mad(ah, w.cl, m);
  n = fx_mad(ah, w.sl, n);
  m = fx_mad(bh, nl, m);
  n = fx_mad(bh, w.cl, n);
  long long re = (long long)ah * w.ch, im = (long long)ah * w.sh;
  re = fx_mad(bh, nh, re);
  im = fx_mad(bh, w.ch, im);
  re = (long long)((unsigned long long)re << 2) + (m >> 30) + half;
  im = (long long)((unsigned long long)im << 2) + (n >> 30) + half;
  return cfx{re >> sh, im >> sh};
}

// ---- conversions ------------------------------------------------------------
constexpr int FX_EMIN = 130;

LM_HD unsigned fx_abs_hi(double d) {
#if defined(__CUDA_ARCH__)
  return (unsigned)__double2hiint(d) & 0x7fffffffu;
#else
  unsigned long long u;
  memcpy(&u, &d, 8);
  return (unsigned)(u >> 32) & 0x7fffffffu;
#endif
}

// d = X 2^(emax - 1081), X truncated; msum accumulates the high words of |X|
LM_HD long long fx_from_double(double d, int emax, unsigned& msum) {
  unsigned long long u;
#if defined(__CUDA_ARCH__)
  u = (unsigned long long)__double_as_longlong(d);
#else
  memcpy(&u, &d, 8);
#endif
  const unsigned hi = (unsigned)(u >> 32), lo = (unsigned)u;
  const int ex = (int)((hi >> 20) & 0x7ffu);
  int k = emax - ex;
  k = k > 63 ? 63 : k;
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;
  const unsigned long long t = (((unsigned long long)mh << 32) | lo) << 6;
  const unsigned long long a = t >> k;
  msum += (unsigned)(a >> 32);
  const long long s = (long long)((int)hi >> 31);
  return ((long long)a ^ s) - s;
}

LM_HD int fx_clz64(unsigned long long a) {
#if defined(__CUDA_ARCH__)
  return __clzll((long long)a);
#else
  return a ? __builtin_clzll(a) : 64;
#endif
}

// X 2^(e - 1081) rounded to nearest, for exponents with 63 < e < 2000
LM_HD double fx_to_double(long long X, int e) {
  const long long s = X >> 63;
  unsigned long long a = (unsigned long long)((X ^ s) - s);
  const int lz = fx_clz64(a);
  a = lz < 64 ? a << lz : 0;
  unsigned long long u = (a >> 11) + ((a >> 10) & 1u) + ((unsigned long long)(unsigned)(e + 4 - lz) << 52);
  u = lz < 64 ? u : 0;
  u |= (unsigned long long)s & 0x8000000000000000ull;
#if defined(__CUDA_ARCH__)
  return __longlong_as_double((long long)u);
#else
  double d;
  memcpy(&d, &u, 8);
  return d;
#endif
}

// total right shift D allowed by the sum bound: ssum = sum over the
// transform of |X| in units of 2^44, rounded up
LM_HD int fx_sum_shift(unsigned ssum) {
#if defined(__CUDA_ARCH__)
  const int n = 32 - __clz((int)ssum);
#else
  const int n = ssum ? 32 - __builtin_clz(ssum) : 0;
#endif
  return n > 15 ? n - 15 : 0;
}
// one thread's contribution to ssum from its 16 components' high words
LM_HD unsigned fx_sum_units(unsigned msum) { return ((msum + 16u) >> 12) + 1u; }

// Pass sequence shared by the kernels (block_fft, gfft) and the host
// table builder: radix-8 passes, then one radix-4 or radix-2 pass for the
// remaining bits.
__host__ __device__ __forceinline__ int fft_num_passes(int log2N) { return (log2N + 2) / 3; }
__host__ __device__ __forceinline__ int fft_pass_lr(int log2N, int p) {
  return p < log2N / 3 ? 3 : log2N % 3;
}

// Host: cos and sin of (pi/4) i/E, 0 <= i <= E = 2^lE, as unsigned fractions of
// 2^64 (1 as 2^64 - 1), by their Taylor series in 128-bit integer products: ten
// terms of at most a unit's error each, so within 2^-60.  (Extended-precision
// library calls are emulated, and slow, on some hosts.)
inline void octant_fx(int i, int lE, unsigned long long& c, unsigned long long& s) {
  typedef unsigned __int128 u128;
  const unsigned long long pi4 = 0xC90FDAA22168C234ull;  // pi/4 2^64
  const unsigned long long a = (unsigned long long)(((u128)pi4 * (unsigned)i) >> lE);
  const unsigned long long a2 = (unsigned long long)(((u128)a * a) >> 64);
  u128 one = (u128)1 << 64, cs = one, sn = a, tc = one, ts = a;
  for (int n = 1; n <= 11; ++n) {
    tc = ((tc * a2) >> 64) / (unsigned)((2 * n - 1) * (2 * n));
    ts = ((ts * a2) >> 64) / (unsigned)((2 * n) * (2 * n + 1));
    if (n & 1) {
      cs -= tc;
      sn -= ts;
    } else {
      cs += tc;
      sn += ts;
    }
  }
  c = cs >= one ? ~0ull : (unsigned long long)cs;
  s = (unsigned long long)sn;
}

// Host: the same table in the fixed-point form of the FP64 group transforms
// (N entries; the last is unused).  Angles are folded into the first octant.
inline void fft_twiddle_table_fx(int log2N, TwFx* tw) {
  const int N = 1 << log2N, E = N / 8;
  std::vector<TwFx> oct(E + 1);
  auto split = [](unsigned long long v, int& h, int& l) {
    // v 2^-64 = h 2^-30 + l 2^-62
    const unsigned long long u = (v >> 2) + ((v >> 1) & 1);
    l = (int)(unsigned)u;
    h = (int)((u >> 32) + ((unsigned)u >> 31));
    if (l == -2147483647 - 1) l = -2147483647;  // negated in places
  };
  for (int i = 0; i <= E; ++i) {
    unsigned long long c, s;
    octant_fx(i, log2N - 3, c, s);
    split(c, oct[i].ch, oct[i].cl);
    split(s, oct[i].sh, oct[i].sl);
  }
  // exp(-2 pi i n/N)
  auto entry = [&](int n) {
    const int q = n / (N / 4), m = n % (N / 4);
    const bool fold = m > E;
    TwFx t = oct[fold ? N / 4 - m : m];
    if (fold) t = TwFx{t.sh, t.sl, t.ch, t.cl};
    // cos, sin of the first-quadrant angle, turned by q quarters, conjugated
    switch (q) {
      case 0: return TwFx{t.ch, t.cl, -t.sh, -t.sl};
      case 1: return TwFx{-t.sh, -t.sl, -t.ch, -t.cl};
      case 2: return TwFx{-t.ch, -t.cl, t.sh, t.sl};
      default: return TwFx{t.sh, t.sl, t.ch, t.cl};
    }
  };
  tw[N - 1] = entry(0);
  int lNs = 0;
  for (int p = 0; p < fft_num_passes(log2N); ++p) {
    const int lr = fft_pass_lr(log2N, p);
    const int Ns = 1 << lNs, R = 1 << lr;
    for (int r = 1; r < R; ++r)
      for (int k = 0; k < Ns; ++k) tw[r * Ns + k - 1] = entry(r * k * (N / (Ns * R)));
    lNs += lr;
  }
}

// Twiddle type of the group transforms.
template <typename T> struct TwidT;
template <> struct TwidT<float> { typedef float2 type; };
template <> struct TwidT<double> { typedef TwFx type; };
template <typename T> using twid = typename TwidT<T>::type;

}  // namespace lm
