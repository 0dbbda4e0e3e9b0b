// kernels.cuh -- what the stage kernels (stage.cuh) are built from, and the
// transforms around the stepping.
//
// One RK stage of the coupled shallow-water + Lagrangian-mean system is
//   row_prod   mixed fields -> products       (inverse x-FFT, physical-space
//              products of the shallow-water equations and of the
//              Lagrangian-mean PDEs, forward x-FFT)
//   col_stage  products -> next mixed fields  (forward y-FFT and 2/3 mask,
//              right-hand sides and the integrating-factor combination,
//              derivatives and inverse y-FFT)
// (Strategy 2, and FP64 from 1024^2, add row_inv into physical planes before
// row_prod.)  The dealiased pseudospectral method is the one the paper uses for
// both the dynamics and the mean equations (Sec. 4.1, 4.2).
#pragma once
#include "common.cuh"
#include "fft.cuh"

namespace lm {

// ---------------------------------------------------------------------------
// Column passes on a tile of C = 2^lC consecutive kx columns (kx0 a multiple
// of C, KXP a multiple of C), C*N/8 threads, smem C*col_stride(N, C) complex.  The
// tile's global accesses are C-wide contiguous runs along kx.

// inverse: d = IFFT_y(s), zero-padded outside |ky| <= K.
template <typename T>
__device__ void col_inverse_tile(cplx<T>* buf, const cplx<T>* __restrict__ s, cplx<T>* __restrict__ d, const Geom& g,
                                 int lC, int kx0, const cplx<T>* __restrict__ tw) {
  const int N = g.N, K = g.K, KXP = g.KXP;
  const int C = 1 << lC, bst = col_stride<T>(N, C);
  const int nthr = blockDim.x, tid = threadIdx.x;
  // every element written once: s at n = ky mod N for |ky| <= K, else 0
  for (int e = tid; e < N * C; e += nthr) {
    const int n = e >> lC, c = e & (C - 1);
    const int kx = kx0 + c;
    const int ky = n <= K ? n : n - N;
    cplx<T> v = mk<T>(0, 0);
    if (kx <= K && (n <= K || n >= N - K)) v = s[(long long)(ky + K) * KXP + kx];
    buf[c * bst + sidx<T>(n)] = v;
  }
  __syncthreads();
  block_fft<T, +1>(buf, g.log2N, bst, tw);
  for (int e = tid; e < N * C; e += nthr) {
    const int n = e >> lC, c = e & (C - 1);
    d[(long long)n * KXP + kx0 + c] = buf[c * bst + sidx<T>(n)];
  }
}

// forward: d = FFT_y(s)/N on the rows |ky| <= K (zero for kx > K).
template <typename T>
__device__ void col_forward_tile(cplx<T>* buf, const cplx<T>* __restrict__ s, cplx<T>* __restrict__ d,
                                 const Geom& g, int lC, int kx0, const cplx<T>* __restrict__ tw) {
  const int N = g.N, K = g.K, KXP = g.KXP;
  const int C = 1 << lC, bst = col_stride<T>(N, C);
  const int nthr = blockDim.x, tid = threadIdx.x;
  for (int e = tid; e < N * C; e += nthr) {
    const int n = e >> lC, c = e & (C - 1);
    buf[c * bst + sidx<T>(n)] = s[(long long)n * KXP + kx0 + c];
  }
  __syncthreads();
  block_fft<T, -1>(buf, g.log2N, bst, tw);
  const T inv = (T)1 / (T)N;
  for (int e = tid; e < g.NY * C; e += nthr) {
    const int kyi = e >> lC, c = e & (C - 1);
    const int kx = kx0 + c;
    const int ky = kyi - K;
    cplx<T> v = mk<T>(0, 0);
    if (kx <= K) v = cscale<T>(buf[c * bst + sidx<T>(ky & (N - 1))], inv);
    d[(long long)kyi * KXP + kx] = v;
  }
}

// Column passes of one field: grid KXP/4, 4 columns per block.
template <typename T>
struct ColArgs {
  const cplx<T>* src;  // inverse: spectral; forward: mixed
  cplx<T>* dst;
  const cplx<T>* tw;
  Geom g;
};

template <typename T>
__global__ void __launch_bounds__(1024) k_col_inv(const __grid_constant__ ColArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  col_inverse_tile<T>(reinterpret_cast<cplx<T>*>(smem_raw), a.src, a.dst, a.g, 2, blockIdx.x * 4, a.tw);
}

template <typename T>
__global__ void __launch_bounds__(1024) k_col_fwd(const __grid_constant__ ColArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  col_forward_tile<T>(reinterpret_cast<cplx<T>*>(smem_raw), a.src, a.dst, a.g, 2, blockIdx.x * 4, a.tw);
}

// ---------------------------------------------------------------------------
// Row helpers.  A block owns B consecutive rows; its FFT buffer holds B
// transforms of length N at stride row_stride(N).

// Fill buf with the Hermitian spectrum of real rows whose kx >= 0 halves are the
// mixed field m, then inverse FFT: afterwards the real part of buf[row][x] is the
// row.  The kx = 0 imaginary part is dropped, as a real inverse transform does.
template <typename T>
__device__ void row_inverse(cplx<T>* buf, const cplx<T>* __restrict__ m, int row0, int B, const Geom& g,
                            const cplx<T>* __restrict__ tw) {
  const int N = g.N, K = g.K, KXP = g.KXP;
  const int bst = row_stride<T>(N);
  const int nthr = blockDim.x, tid = threadIdx.x;
  // Z(k) = A and Z(N-k) = conj(A) for k <= K (each input read once); the band
  // K < n < N-K is zeroed.  The two writes never touch the same element, so no
  // barrier separates them.
  const int nz = N - 2 * K - 1;
  for (int e = tid; e < B * nz; e += nthr) {
    const int r = e / nz, n = K + 1 + (e - r * nz);
    buf[r * bst + sidx<T>(n)] = mk<T>(0, 0);
  }
  for (int e = tid; e < B * (K + 1); e += nthr) {
    const int r = e / (K + 1), k = e - r * (K + 1);
    const cplx<T> A = m[(long long)(row0 + r) * KXP + k];
    cplx<T>* z = buf + r * bst;
    if (k == 0) {
      z[0] = mk<T>(A.x, 0);
    } else {
      z[sidx<T>(k)] = A;
      z[sidx<T>(N - k)] = mk<T>(A.x, -A.y);
    }
  }
  __syncthreads();
  block_fft<T, +1>(buf, g.log2N, bst, tw);
}

// Forward FFT of buf (real rows) and store of the kx in [0, KXP) half, scaled by
// 1/N, into the mixed field d.
template <typename T>
__device__ void row_forward_store(cplx<T>* buf, cplx<T>* __restrict__ d, int row0, int B, const Geom& g,
                                  const cplx<T>* __restrict__ tw) {
  const int N = g.N, K = g.K, KXP = g.KXP;
  const int bst = row_stride<T>(N);
  const int nthr = blockDim.x, tid = threadIdx.x;
  __syncthreads();
  block_fft<T, -1>(buf, g.log2N, bst, tw);
  const T h = (T)0.5 / (T)N;
  for (int e = tid; e < B * KXP; e += nthr) {
    const int r = e / KXP, k = e - r * KXP;
    const cplx<T>* z = buf + r * bst;
    cplx<T> P = mk<T>(0, 0);
    if (k <= K) {
      // (Z(k) + conj Z(N-k))/2
      const cplx<T> z1 = z[sidx<T>(k)], z2 = z[sidx<T>((N - k) & (N - 1))];
      P = mk<T>((z1.x + z2.x) * h, (z1.y - z2.y) * h);
    }
    d[(long long)(row0 + r) * KXP + k] = P;
  }
}

// Group-owned row transforms (one row per group of G = N/8 threads, N = 2^L
// fixed at compile time; thread j holds positions j + m G, see gfft).

// Hermitian-paired spectrum of the two real rows of a row pair (A, B: their kx
// >= 0 halves, interleaved at r) at the thread's positions k = j + m G:
// Z(k) = A(k) + i B(k) for k <= K, conj A(N-k) + i conj B(N-k) for k >= N-K,
// zero in between; the kx = 0 imaginary parts are dropped, as a real inverse
// transform does.  Parts are swapped: the inverse transform runs as a forward
// one, and leaves row A in the imaginary and row B in the real part.
template <typename T, int L>
__device__ __forceinline__ void load_rows_ct(cplx<T> (&x)[8], const cplx<T>* r, int j, int K) {
  constexpr int N = 1 << L, G = N / 8;
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    if (m == 3 || m == 4) {  // N/4 <= K < 3N/8: never in the box
      x[m] = mk<T>(0, 0);
      continue;
    }
    const int k = j + m * G;
    const int kk = m < 4 ? k : N - k;
    const bool in = kk <= K;
    cplx<T> A, Bv;
    ld_pair(r + 2 * (in ? kk : 0), A, Bv);
    cplx<T> z;
    if (m < 4) z = mk<T>(A.y + Bv.x, A.x - Bv.y);
    else z = mk<T>(Bv.x - A.y, A.x + Bv.y);
    if (m == 0 && j == 0) z = mk<T>(Bv.x, A.x);
    x[m] = in ? z : mk<T>(0, 0);
  }
}

// Spectrum Z of p + i q (the two rows), times 1/(2 N), held at the thread's
// positions -> kx in [0, K] halves of p and q (times 1/N), interleaved at r.
// One exchange through the free buffer.  (The padding columns kx > K are left as
// they are: a column pass transforms them and drops the result.)
template <typename T, int L, int SYNC>
__device__ __forceinline__ void store_rows_ct(const cplx<T> (&x)[8], cplx<T>* buf0, cplx<T>* buf1, int& w,
                                              cplx<T>* __restrict__ r, int j, int grp, int K) {
  constexpr int N = 1 << L, G = N / 8;
  cplx<T>* b = w ? buf1 : buf0;
  if constexpr (G % 8 == 0) {
    const int sb = j + (j >> 3);
#pragma unroll
    for (int m = 0; m < 8; ++m)
      if (m != 3 && m != 4) b[sb + m * (G + G / 8)] = x[m];  // sidx(j + m G)
  } else {
#pragma unroll
    for (int m = 0; m < 8; ++m) b[sidx<T>(j + m * G)] = x[m];
  }
  gsync<SYNC, G>(grp);
  // K < 3 G
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int k = j + i * G;
    if (k <= K) {
      const cplx<T> z1 = b[k + (k >> 3)];
      const int k2 = (N - k) & (N - 1);
      const cplx<T> z2 = b[k2 + (k2 >> 3)];
      // P = Z(k) + conj Z(N-k), Q = (Z(k) - conj Z(N-k))/i
      st_pair(r + 2 * k, mk<T>(z1.x + z2.x, z1.y - z2.y), mk<T>(z1.y + z2.y, z2.x - z1.x));
    }
  }
  w ^= 1;
}

// Call f(IntC<L>()) for the run-time length exponent L in [LO, HI]: the
// stage kernels' bodies are compiled once per transform length.
template <int V> struct IntC { static constexpr int value = V; };
template <int LO, int HI, typename F>
__device__ __forceinline__ void dispatch_L(int L, F&& f) {
  if constexpr (LO <= HI) {
    if (L == LO) f(IntC<LO>());
    else dispatch_L<LO + 1, HI>(L, f);
  }
}

// ---------------------------------------------------------------------------
// Row passes of one field between mixed rows and FP64 physical rows, B rows per
// block.
template <typename T, typename S, typename D>
struct RowArgs {
  const S* src;
  D* dst;
  const cplx<T>* tw;
  Geom g;
  int B;
};
template <typename T> using RowInvArgs = RowArgs<T, cplx<T>, double>;
template <typename T> using RowFwdArgs = RowArgs<T, double, cplx<T>>;

template <typename T>
__global__ void __launch_bounds__(256) k_row_inv(const __grid_constant__ RowInvArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cplx<T>* buf = reinterpret_cast<cplx<T>*>(smem_raw);
  const int N = a.g.N, B = a.B, row0 = blockIdx.x * B;
  row_inverse<T>(buf, a.src, row0, B, a.g, a.tw);
  for (int e = threadIdx.x; e < B * N; e += blockDim.x) {
    const int r = e / N, x = e - r * N;
    a.dst[(long long)(row0 + r) * N + x] = (double)buf[r * row_stride<T>(N) + sidx<T>(x)].x;
  }
}

template <typename T>
__global__ void __launch_bounds__(256) k_row_fwd(const __grid_constant__ RowFwdArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cplx<T>* buf = reinterpret_cast<cplx<T>*>(smem_raw);
  const int N = a.g.N, B = a.B, row0 = blockIdx.x * B;
  for (int e = threadIdx.x; e < B * N; e += blockDim.x) {
    const int r = e / N, x = e - r * N;
    buf[r * row_stride<T>(N) + sidx<T>(x)] = mk<T>((T)a.src[(long long)(row0 + r) * N + x], (T)0);
  }
  row_forward_store<T>(buf, a.dst, row0, B, a.g, a.tw);
}

// ---------------------------------------------------------------------------
// Interval time of a stage: s = (steps done + c_stage) * dt, from the device
// step counter (never accumulated).
// time of a stage in steps: RK4 (0, 1/2, 1/2, 1), Heun (0, 1), Euler (0)
// Computed in the kernel's precision T: sm_103 issues FP64 arithmetic at a
// small fraction of the FP32 rate, so FP32 kernels keep it out of the set-up
// every thread runs.
// The 64-bit step count is converted through its two 31-bit halves (exact
// in FP64 below 2^53 steps, and in FP32 below 2^24).
template <typename T>
__device__ __forceinline__ T stage_time(long long n, int stage, T dt, int stepper) {
  const T steps = (T)(int)(n >> 31) * (T)2147483648.0 + (T)(int)(n & 0x7fffffffLL);
  const T c = stage == 0 ? (T)0 : (stepper != 0 || stage == 3 ? (T)1 : (T)0.5);
  return (steps + c) * dt;
}

// Bilinear interpolation of the periodic grid fields at (x_i + xi_x, y_j + xi_y)
// (Sec. 4.2.1): corner offsets and weights.  The displacement in cells d =
// xi/dx gives the cell index i + floor(d) and the weight d - floor(d).  Indices
// wrap with & (N-1), so any displacement (even a non-finite one) reads inside
// the field.
template <typename T> struct Bilin {
  unsigned o00, o01, o10, o11;
  T w00, w01, w10, w11;
  __device__ __forceinline__ Bilin(int i, int j, T xi_x, T xi_y, T inv_dx, int N) {
    const T dxc = mul_rn(xi_x, inv_dx), dyc = mul_rn(xi_y, inv_dx);
    unsigned kx, ky;
    const T fx = floor_int(dxc, kx), fy = floor_int(dyc, ky);
    const T ax = dxc - fx, ay = dyc - fy;
    const unsigned msk = (unsigned)N - 1u;
    const unsigned i0 = ((unsigned)i + kx) & msk;
    const unsigned j0 = ((unsigned)j + ky) & msk;
    const unsigned i1 = (i0 + 1u) & msk, j1 = (j0 + 1u) & msk;
    o00 = j0 * N + i0;
    o01 = j0 * N + i1;
    o10 = j1 * N + i0;
    o11 = j1 * N + i1;
    w00 = ((T)1 - ax) * ((T)1 - ay);
    w01 = ax * ((T)1 - ay);
    w10 = ((T)1 - ax) * ay;
    w11 = ax * ay;
  }
};
template <typename T>
__device__ __forceinline__ T bilinear(const T* f, int i, int j, T xi_x, T xi_y, T inv_dx, int N) {
  const Bilin<T> b(i, j, xi_x, xi_y, inv_dx, N);
  return fma(b.w11, gld(f + b.o11), fma(b.w10, gld(f + b.o10), fma(b.w01, gld(f + b.o01), mul_rn(b.w00, gld(f + b.o00)))));
}
__device__ __forceinline__ void ld_quad(const float* p, float* v) {
  const float4 q = gld(reinterpret_cast<const float4*>(p));
  v[0] = q.x;
  v[1] = q.y;
  v[2] = q.z;
  v[3] = q.w;
}
__device__ __forceinline__ void ld_quad(const double* p, double* v) {
  const double2 a = gld(reinterpret_cast<const double2*>(p)), b = gld(reinterpret_cast<const double2*>(p) + 1);
  v[0] = a.x;
  v[1] = a.y;
  v[2] = b.x;
  v[3] = b.y;
}

// ---------------------------------------------------------------------------
// Two-dimensional Euler model: u, v of the vorticity in slot fh, through the
// streamfunction (u_hat = i ky zeta_hat/|k|^2, v_hat = -i kx zeta_hat/|k|^2,
// zero at k = 0), into slots fu, fv; one thread per box mode.
template <typename T>
__global__ void k_velocity_from_vorticity(cplx<T>* __restrict__ y, Geom g, int fu, int fv, int fh) {
  const long long m = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= g.ms) return;
  const int mi = (int)m;
  const int kyi = mi / g.KXP, kx = mi - kyi * g.KXP;
  const T kxf = (T)kx, kyf = (T)(kyi - g.K);
  const int o = spec_index<T>(kyi, kx, g.NY);
  const cplx<T> z = y[(long long)fh * g.ms + o];
  const T k2 = kxf * kxf + kyf * kyf;
  const T inv = k2 > (T)0 ? (T)1 / k2 : (T)0;
  y[(long long)fu * g.ms + o] = mk<T>(-kyf * z.y * inv, kyf * z.x * inv);
  y[(long long)fv * g.ms + o] = mk<T>(kxf * z.y * inv, -kxf * z.x * inv);
}

// ---------------------------------------------------------------------------
// FP64 transforms around the stepping (initial conditions, results), on the
// fixed-point group transforms.  A launch takes up to four fields: a column
// pass between the state (tile-blocked, in T) and FP64 mixed fields
// (interleaved row pairs), and a row pass between these and FP64 physical
// planes.  (As one FP64-butterfly launch each for a conversion, a column and a
// row pass per pair of fields, u, v, h and zeta took nine launches; a
// semi-Lagrangian step at 256^2, which needs them, 232 us, now 126 us.)
constexpr int IO_MAX = 4;
// Columns per block: as the column stage in FP64.
__host__ __device__ __forceinline__ int io_log2C(int N) {
  int l = 0;
  while ((N << l) < 256 || ((N << l) < 2 * N && N < 2048)) ++l;
  return l;
}

template <typename T> struct OutArgs {
  const cplx<T>* y;
  const cplx<T>* comp;  // compensation terms to subtract (null: none)
  double2* mix;
  double* phys;
  const TwFx* tw;
  Geom g;
  int n;
  int field[IO_MAX], field2[IO_MAX];  // field2 >= 0: i kx field2 - i ky field
  int slot[IO_MAX];                   // plane of phys
  // value = scale*val + ax*x + ay*y + cst
  double scale[IO_MAX], ax[IO_MAX], ay[IO_MAX], cst[IO_MAX];
};

// Local block = (field, kx tile).
template <typename T>
__global__ void __launch_bounds__(256) k_out_col(const __grid_constant__ OutArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned red[GRED_WORDS];
  dispatch_L<4, 11>(a.g.log2N, [&](auto Lc) {
    constexpr int L = decltype(Lc)::value, N = 1 << L, G = N / 8, CS = spec_tile<T>();
    const int lC = io_log2C(N), C = 1 << lC;
    const int i = blockIdx.y, c = threadIdx.x & (C - 1), j = threadIdx.x >> lC;
    const int kx = (blockIdx.x << lC) + c, K = a.g.K, KXP = a.g.KXP, ms = (int)a.g.ms;
    const int m00 = (kx / CS) * (a.g.NY * CS) + kx % CS;
    double2 x[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int n = j + m * G, ky = n <= K ? n : n - N;
      x[m] = make_double2(0.0, 0.0);
      if (kx <= K && ky >= -K) {
        const int o = (ky + K) * CS + m00;
        auto val = [&](int f) {
          const cplx<T> v = a.y[f * ms + o];
          double2 r = make_double2((double)v.x, (double)v.y);
          if (a.comp) {
            const cplx<T> q = a.comp[f * ms + o];
            r.x -= (double)q.x;
            r.y -= (double)q.y;
          }
          return r;
        };
        x[m] = val(a.field[i]);
        if (a.field2[i] >= 0)
          x[m] = csub<double>(cik<double>(val(a.field2[i]), (double)kx), cik<double>(x[m], (double)ky));
      }
    }
    double2* b0 = reinterpret_cast<double2*>(smem_raw) + (size_t)c * col_buf_stride<double>(N, C);
    int w = 0;
    gfft<double, +1, L, 2>(x, b0, b0 + row_stride<double>(N), w, j, 0, a.tw, GRed{red, lC, (int)threadIdx.x, (int)blockDim.x});
    double2* dst = a.mix + (long long)i * a.g.mi + (j >> 1) * 2 * KXP + 2 * kx + (j & 1);
#pragma unroll
    for (int m = 0; m < 8; ++m) dst[m * G * KXP] = x[m];
  });
}

// Local block = (field, block of row pairs, one per group of N/8 threads).
template <typename T>
__global__ void __launch_bounds__(256) k_out_row(const __grid_constant__ OutArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned red[GRED_WORDS];
  dispatch_L<4, 11>(a.g.log2N, [&](auto Lc) {
    constexpr int L = decltype(Lc)::value, N = 1 << L, G = N / 8, SYNC = L <= 8 ? 0 : 1;
    constexpr int rs = N + N / 8;
    const int i = blockIdx.y, gi = threadIdx.x / G, j = threadIdx.x - gi * G;
    const int yp = (blockIdx.x * (blockDim.x / G) + gi) & (N / 2 - 1);
    double2* buf0 = reinterpret_cast<double2*>(smem_raw) + (size_t)gi * 2 * rs;
    double2 x[8];
    int w = 0;
    load_rows_ct<double, L>(x, a.mix + (long long)i * a.g.mi + (long long)yp * 2 * a.g.KXP, j, a.g.K);
    gfft<double, -1, L, SYNC>(x, buf0, buf0 + rs, w, j, gi, a.tw, GRed{red, 0, 0, 0});
    const double dxg = 6.283185307179586476925286766559 / (double)N;
    const double s = a.scale[i], ax = a.ax[i], ay = a.ay[i], cst = a.cst[i];
    double* p = a.phys + (long long)a.slot[i] * a.g.np + (long long)yp * 2 * N + j;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const double xg = ax * ((j + m * G) * dxg);
      p[m * G] = s * x[m].y + xg + ay * ((2 * yp) * dxg) + cst;
      p[N + m * G] = s * x[m].x + xg + ay * ((2 * yp + 1) * dxg) + cst;
    }
  });
}

template <typename T> struct InArgs {
  const double* phys;
  double2* mix;
  cplx<T>* y;
  const TwFx* tw;
  Geom g;
  int n;
  int slot[IO_MAX], field[IO_MAX];
  double mean[IO_MAX];  // added to the k = 0 coefficient
};

template <typename T>
__global__ void __launch_bounds__(256) k_in_row(const __grid_constant__ InArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned red[GRED_WORDS];
  dispatch_L<4, 11>(a.g.log2N, [&](auto Lc) {
    constexpr int L = decltype(Lc)::value, N = 1 << L, G = N / 8, SYNC = L <= 8 ? 0 : 1;
    constexpr int rs = N + N / 8;
    const int i = blockIdx.y, gi = threadIdx.x / G, j = threadIdx.x - gi * G;
    const int yp = (blockIdx.x * (blockDim.x / G) + gi) & (N / 2 - 1);
    double2* buf0 = reinterpret_cast<double2*>(smem_raw) + (size_t)gi * 2 * rs;
    const double* p = a.phys + (long long)a.slot[i] * a.g.np + (long long)yp * 2 * N + j;
    double2 x[8];
    int w = 0;
#pragma unroll
    for (int m = 0; m < 8; ++m) x[m] = make_double2(p[m * G], p[N + m * G]);
    gfft<double, -1, L, SYNC>(x, buf0, buf0 + rs, w, j, gi, a.tw, GRed{red, 0, 0, 0}, -L - 1);
    store_rows_ct<double, L, SYNC>(x, buf0, buf0 + rs, w, a.mix + (long long)i * a.g.mi + (long long)yp * 2 * a.g.KXP,
                                   j, gi, a.g.K);
  });
}

template <typename T>
__global__ void __launch_bounds__(256) k_in_col(const __grid_constant__ InArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned red[GRED_WORDS];
  dispatch_L<4, 11>(a.g.log2N, [&](auto Lc) {
    constexpr int L = decltype(Lc)::value, N = 1 << L, G = N / 8, CS = spec_tile<T>();
    const int lC = io_log2C(N), C = 1 << lC;
    const int i = blockIdx.y, c = threadIdx.x & (C - 1), j = threadIdx.x >> lC;
    const int kx = (blockIdx.x << lC) + c, K = a.g.K, KXP = a.g.KXP;
    const double2* src = a.mix + (long long)i * a.g.mi + (j >> 1) * 2 * KXP + 2 * kx + (j & 1);
    double2 x[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) x[m] = src[m * G * KXP];
    double2* b0 = reinterpret_cast<double2*>(smem_raw) + (size_t)c * col_buf_stride<double>(N, C);
    int w = 0;
    gfft<double, -1, L, 2>(x, b0, b0 + row_stride<double>(N), w, j, 0, a.tw, GRed{red, lC, (int)threadIdx.x, (int)blockDim.x},
                           -L);
    cplx<T>* dst = a.y + (long long)a.field[i] * a.g.ms + (kx / CS) * (a.g.NY * CS) + kx % CS;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int n = j + m * G, ky = n <= K ? n : n - N;
      if (ky < -K) continue;
      if (n == 0 && kx == 0) x[m].x += a.mean[i];
      dst[(ky + K) * CS] = kx <= K ? mk<T>((T)x[m].x, (T)x[m].y) : mk<T>((T)0, (T)0);
    }
  });
}

// Copy of nf fields of the state (t0) and of their compensation terms (t1)
// between the tile-blocked layout and rows [ky + K][kx] (checkpoint blobs: the
// fields of t0, then those of t1); to_rows: rows get the copy, else the step
// counter ctr is set to `done` too.
template <typename T>
__global__ void k_spec_rows(cplx<T>* __restrict__ t0, cplx<T>* __restrict__ t1, cplx<T>* __restrict__ rows, Geom g,
                            int nf, int to_rows, long long* ctr, long long done) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0 && !to_rows) *ctr = done;
  if (i >= g.ms * 2 * nf) return;
  const int f = (int)(i / g.ms), m = (int)(i - f * g.ms);
  cplx<T>* t = (f < nf ? t0 + f * g.ms : t1 + (f - nf) * g.ms) + spec_index<T>(m / g.KXP, m % g.KXP, g.NY);
  if (to_rows) rows[i] = *t;
  else *t = rows[i];
}

// ---------------------------------------------------------------------------
// Deterministic FP64 invariant sums over a physical grid (u, v, h, zeta):
// per-block partial sums, then one block adds the partials in fixed order.
__global__ void k_diag_partial(const double* __restrict__ phys, long long np, double f0, double c2,
                               double* __restrict__ part);
__global__ void k_diag_final(const double* __restrict__ part, int nblk, long long np, double* __restrict__ out);

}  // namespace lm
