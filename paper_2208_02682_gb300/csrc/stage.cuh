// stage.cuh -- the kernels of one RK stage, over a batch of independent runs.
//
// Every stage kernel takes a device table of run descriptors and, per kernel
// kind, a prefix sum of the blocks each run needs: block b belongs to the run
// r with start[r] <= b < start[r+1] and works on local block b - start[r].
// A single handle is a batch of one; sw_batch steps many handles (different
// grid sizes, strategies and field sets) in the same launches.  Block shapes
// are uniform within a launch: C*N (columns x points) and Bp*N, Bi*N (rows x
// points) are equal for all members.
//
// Per stage:  [row_inv] -> row_prod -> col_stage [-> kin, for runs without
// transforms]; a replay of steps starts with one col_stage that only transforms.
#pragma once
#include "kernels.cuh"

namespace lm {

enum { KT_ROW_INV = 0, KT_ROW_PROD = 1, KT_COL_STAGE = 2, KT_KIN = 3, KT_COUNT = 4 };

template <typename T>
struct alignas(16) RunDesc {
  Geom g;
  Layout L;
  StepConsts c;
  T cdt, cf0, cc2, cadvx, cadvy;  // dt, f0, c2, adv in the kernels' precision
  T cci;          // weight of the summed right-hand sides in the commit: dt/6, dt/2 or 1 (by stepper)
  cplx<T>* y;     // state at t_n
  cplx<T>* ysa;   // stage inputs of stages 1 and 3 (u, v, h)
  cplx<T>* ysb;   // stage input of stage 2 (u, v, h)
  cplx<T>* acc;   // RK accumulator
  cplx<T>* comp;  // Kahan compensation (FP32 mode; null in FP64)
  cplx<T>* mix;   // column-pass outputs (mixed)
  cplx<T>* pmix;  // row-pass products (mixed)
  T* phys;        // Strategy-2 gather buffer
  const T* ef;    // integrating-factor tables
  const twid<T>* tw;
  long long* ctr;
  unsigned* ticket;
  int lC;         // column tile: C = 2^lC columns
  int Bp, ppb;    // row_prod: row pairs per block, products per block
  int Wp;         // row_prod: groups of N/8 threads per row pair
  int team;       // row_inv, row_prod: a team of four sets of groups per row pair
  int hzsep;      // row_inv: zeta in blocks of its own
  int Bi;         // row_inv: row pairs per block
  int fused;      // row_prod: transforms the base fields itself
  int gath;       // row_prod: gathers all fields at x + xi at once (interleaved planes)
  int umask[MAXP];  // row_prod: base fields each product chunk needs (bits PH_*)
  int nb[KT_COUNT];
};

__device__ __forceinline__ int find_run(const int* __restrict__ start, int nruns, int b) {
  int lo = 0, hi = nruns;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (start[mid] <= b) lo = mid;
    else hi = mid;
  }
  return lo;
}

// Copy the block's run descriptor into shared memory with one cooperative
// load, so the kernel's many field-index and pointer lookups are shared-memory
// reads instead of chains of dependent global loads.
template <typename T>
__device__ __forceinline__ const RunDesc<T>& load_desc(const RunDesc<T>* __restrict__ runs, int r,
                                                       unsigned char* sbuf) {
  static_assert(sizeof(RunDesc<T>) % sizeof(int4) == 0, "descriptor size");
  const int4* src = reinterpret_cast<const int4*>(runs + r);
  int4* dst = reinterpret_cast<int4*>(sbuf);
  constexpr int n = (int)(sizeof(RunDesc<T>) / sizeof(int4));
#pragma unroll 4
  for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = __ldg(src + i);
  __syncthreads();
  return *reinterpret_cast<const RunDesc<T>*>(sbuf);
}

#define LM_STAGE_DESC(T_)                                                 \
  __shared__ __align__(16) unsigned char sdesc_[sizeof(RunDesc<T_>)];   \
  const RunDesc<T_>& d = load_desc<T_>(runs, r, sdesc_)

template <typename T>
__device__ __forceinline__ const cplx<T>* stage_input(const RunDesc<T>& d, int stage) {
  return stage == 0 ? d.y : (stage == 2 ? d.ysb : d.ysa);
}

// a3: base planes (physical u, v, h, zeta and, Strategy 2, xi and, with PV
// averaged, q = (f0 + zeta)/h, h = 1 + eta) of the runs whose row pass does not
// form them itself.  Local block = (field, block of Bi row pairs, one pair per
// group of N/8 threads); a team's block has four sets of groups, of which h, zeta and q
// use more than one (16^2 FP64: 12.3 -> 10.5 us, with q 18.4 -> 12.4).
template <typename T, bool WARP>
__global__ void __launch_bounds__(256) k_stage_row_inv(const RunDesc<T>* __restrict__ runs,
                                                       const int* __restrict__ start, int nruns) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned red[GRedWords<T>::value];  // FP64 transforms
  const int r = find_run(start, nruns, blockIdx.x);
  const RunDesc<T>& d = runs[r];
  pdl_wait();  // state written by the previous kernels: only after this
  pdl_release();
  const int lb = blockIdx.x - start[r];
  auto body = [&](auto Lc) {
    constexpr int L = decltype(Lc)::value, N = 1 << L, G = N / 8;
    constexpr int SYNC = L <= 8 ? 0 : 1;
    const Geom& g = d.g;
    const int B = d.Bi;
    const int nrb = max(N / 2 / B, 1);
    const int f = lb / nrb, rb = lb - f * nrb;
    const int grp = threadIdx.x / G, j = threadIdx.x - grp * G;
    const bool team = G < 32 && d.team != 0;
    const int set = team ? grp / B : 0, row = grp - set * B;
    const int yp = (rb * B + row) & (N / 2 - 1);
    constexpr int rs = N + N / 8;
    cplx<T>* buf0 = reinterpret_cast<cplx<T>*>(smem_raw) + (size_t)grp * 2 * rs;
    cplx<T> x[8], eta[8];
    int w = 0;
    // the field of h takes zeta too, unless zeta has blocks of its own (the last)
    const bool hz = f == 2 && !d.hzsep, zl = f == (d.L.strategy == 2 ? 5 : 3);
#pragma unroll 1
    for (int part = set; part < (hz ? (set ? 2 : (team ? 1 : 2)) : 1); ++part) {
      const bool z = zl || (hz && part);
      const int src = z ? d.L.i_z : (f == 0 ? d.L.i_u : (f == 1 ? d.L.i_v : (f == 2 ? d.L.i_h : d.L.i_xi[f - 3])));
      const int dst = z ? PH_Z : (f <= PH_H ? f : f - 3 + PH_XX);
      load_rows_ct<T, L>(x, d.mix + (long long)src * g.mi + (long long)yp * 2 * g.KXP, j, g.K);
      gfft<T, -1, L, SYNC>(x, buf0, buf0 + rs, w, j, grp, d.tw, GRed{red, 0, 0, 0});
      // planes [y][x]; interleaved, the four base fields as [y][x][4] and the
      // two components of xi as [y][x][2]
      const int es = !d.gath ? 1 : (dst < 4 ? 4 : 2);
      T* p = d.phys + (long long)(es == 1 ? dst : (es == 4 ? 0 : PH_XX)) * g.np +
             (es == 1 ? 0 : (es == 4 ? dst : dst - PH_XX)) + ((long long)yp * 2 * N + j) * es;
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        p[m * G * es] = x[m].y;
        p[(N + m * G) * es] = x[m].x;
      }
      if (part == 0) {
#pragma unroll
        for (int m = 0; m < 8; ++m) eta[m] = x[m];
      }
    }
    if (team && hz && d.L.has_q) {
      // eta and zeta to the four sets, two of the eight positions each
      cplx<T>* E = reinterpret_cast<cplx<T>*>(smem_raw) + (size_t)(2 * B + row) * 2 * rs + j;
      cplx<T>* Z = E + (size_t)B * 2 * rs;
      if (set < 2) {
#pragma unroll
        for (int m = 0; m < 8; ++m) (set ? Z : E)[m * G] = x[m];
      }
      __syncthreads();
      T* p = d.phys + (long long)PH_Q * g.np + (long long)yp * 2 * N + j;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int m = 2 * set + i;
        const cplx<T> z = Z[m * G], e = E[m * G];
        p[m * G] = (d.cf0 + z.y) / ((T)1 + e.y);
        p[N + m * G] = (d.cf0 + z.x) / ((T)1 + e.x);
      }
    } else if (hz && d.L.has_q) {
      T* p = d.phys + (long long)PH_Q * g.np + (long long)yp * 2 * N + j;
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        p[m * G] = (d.cf0 + x[m].y) / ((T)1 + eta[m].y);
        p[N + m * G] = (d.cf0 + x[m].x) / ((T)1 + eta[m].x);
      }
    }
  };
  if constexpr (WARP) dispatch_L<4, 8>(d.g.log2N, body);
  else dispatch_L<4, 11>(d.g.log2N, body);
}

// ---------------------------------------------------------------------------
// a2: row pass with products, on pairs of rows: a complex transform carries
// row 2y as its real and row 2y + 1 as its imaginary part, so that one 16-byte
// (FP32) access of the row-interleaved mixed layout feeds both, and products
// are formed for the two rows at once.  (Pairing two fields of one row, as an
// earlier form did, moved 8 bytes per access and tied products together.)
//
// Local block = (product chunk, block of Bp row pairs): Wp groups of G = N/8
// threads per pair share out the chunk's ppb products, the costly ones first.
// `fused` runs (Strategy 1, except in FP64 from 1024^2): the groups first
// transform the pair's base fields u, v, h, zeta (those the chunk needs) into
// shared memory.  The others read base values from the planes that the row
// inverse pass wrote; Strategy 2 gathers from them too: `gath` runs (where the
// arrays fit and a block takes all products) once for all products, into shared
// memory, from interleaved planes (each product gathering for itself from
// separate planes took 34.7 us at 512^2 with five means, this 26.7 us).  Every transform stays in the
// registers of its group: an advection product takes the inverse transforms
// of d_x G and d_y G and, from the same positions, the forward transform of
// u d_x G + v d_y G; one transform instance serves both directions (the
// inverse as a forward transform of swapped parts), which keeps the code
// within the instruction caches.
// Groups that do different numbers of transforms never share a warp barrier:
// Wp > 1 only when a group is a whole number of warps (N >= 256), or for a `team`.
// Team: while a small grid (N <= 128) leaves most of the GPU idle a launch is as long
// as one block's chain of dependent transforms and of the pointwise work of a lone
// warp (in FP64 64 clocks an instruction), so a block takes one product with four
// sets of groups, a warp or more each: the base fields side by side, then set 0 d_x and
// the forward transform, set 1 d_y, sets 2 and 3 (Strategy 2) the gather of a row each.
// An advection product's chain is three transforms instead of five, a Strategy-2
// product's two instead of three and the gather (16^2 FP64 alone: 34 -> 17.5 us).
// Smem: per pair row_prod_planes() arrays of N complex (fused: the base
// fields; gath: these, xi and the fields at x + xi); per group two
// exchange buffers of row_stride(N) complex.

// Threads per row-pass block at most: three groups at 2048^2 (FP32, 85
// registers), 256 in FP64.
template <typename T> constexpr int row_prod_max_threads() { return sizeof(T) == 4 ? 768 : 256; }

// Arrays of a row pair in shared memory.
__host__ __device__ __forceinline__ int row_prod_planes(int fused, int gath, int has_q) {
  return fused ? 4 : (gath ? 10 + (has_q ? 1 : 0) : 0);
}

__device__ __forceinline__ bool product_heavy(int k) { return k == PK_ADV || k == PK_XI || k == PK_GBAR; }

template <typename T, bool WARP>
__global__ void __launch_bounds__(row_prod_max_threads<T>(), sizeof(T) == 4 ? 1 : 2)
    k_stage_row_prod(const RunDesc<T>* __restrict__ runs, const int* __restrict__ start, int nruns, int stage) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned red[GRedWords<T>::value];  // FP64 transforms
  const int r = find_run(start, nruns, blockIdx.x);
  LM_STAGE_DESC(T);  // field and product lookups from shared memory
  pdl_wait();  // state written by the previous kernels: only after this
  pdl_release();
  const int lb = blockIdx.x - start[r];
  auto body = [&](auto Lc) {
    constexpr int L_ = decltype(Lc)::value, N = 1 << L_, G = N / 8;
    constexpr int SYNC = L_ <= 8 ? 0 : 1;
    constexpr int rs = N + N / 8;
    const Geom& g = d.g;
    const Layout& L = d.L;
    const int B = d.Bp, W = d.Wp, ppb = d.ppb;
    const int nrb = max(N / 2 / B, 1);
    const int pg = lb / nrb, rb = lb - pg * nrb;
    const int gi = threadIdx.x / G, j = threadIdx.x - gi * G;
    // sets of groups: whole warps each for a team, neighbours otherwise
    const bool team = G < 32 && d.team != 0;
    int row = gi / W, wg = gi - row * W;
    if (team) {
      wg = gi / B;
      row = gi - wg * B;
    }
    const int yp = (rb * B + row) & (N / 2 - 1);  // row pair (2 yp, 2 yp + 1)
    const bool fused = d.fused != 0, gath = d.gath != 0, kin = L.model == 1;
    const int nu = row_prod_planes(d.fused, d.gath, L.has_q);
    cplx<T>* U = reinterpret_cast<cplx<T>*>(smem_raw) + (size_t)row * nu * N + j;
    cplx<T>* buf0 = reinterpret_cast<cplx<T>*>(smem_raw) + (size_t)B * nu * N + (size_t)gi * 2 * rs;
    cplx<T>* buf1 = buf0 + rs;
    const int p0 = pg * ppb, p1 = min(L.np, p0 + ppb);
    const T adv_x = d.cadvx, adv_y = d.cadvy, f0 = d.cf0;
    // Strategy 2: the interval time s (the others skip its conversions and
    // divisions in FP64, where they are slow)
    const bool xf = L.scheme == SCHEME_XI_FIRST;
    bool s0 = true;
    T inv_s = (T)0, inv_sg = (T)0;
    if (sizeof(T) == 4 || L.strategy == 2) {
      const T s = stage_time<T>(*d.ctr, stage, d.cdt, d.c.stepper);
      s0 = !(s > (T)0);
      if (!s0) inv_s = (T)1 / s;
      // xi-first scheme: gbar steps with the updated xi at its time s + dt
      inv_sg = xf ? (T)1 / (s + d.cdt) : inv_s;
    }
    const T inv_dx = (T)N / (T)6.283185307179586476925286766559;
    const cplx<T>* mix = d.mix + (long long)yp * 2 * g.KXP;
    const T* phys = d.phys;
    const int rowoff = yp * 2 * N + j;
    const GRed gr = {red, 0};
    int w = 0;
    cplx<T> x[8], acc[8];
    // base field f (PH_*) of both rows at the thread's position m
    auto base = [&](int f, int m) {
      if (fused || gath) return U[(f < 4 ? f : f - 1) * N + m * G];
      const T* p = phys + (long long)f * g.np + rowoff + m * G;
      return mk<T>(gld(p), gld(p + N));
    };

    if (gath) {
      // Strategy 2: the pair's base fields and xi, and the fields at x + xi
      // (Eqs. xi_evol, barf_xi; bilinear interpolation) into shared memory,
      // the points shared out over the pair's threads: one 4-field access per
      // corner serves every product
      T* S = reinterpret_cast<T*>(U - j);
      const T* Q = phys + (long long)PH_Q * g.np;
      for (int e = wg * G + j; e < 2 * N; e += W * G) {
        const int rr = e >= N ? 1 : 0, xcol = e - rr * N, y = 2 * yp + rr;
        const int o = y * N + xcol;
        T b[4], xi[2], f[4];
        ld_quad(phys + 4 * (long long)o, b);
        const cplx<T> xv = gld(reinterpret_cast<const cplx<T>*>(phys + (long long)PH_XX * g.np) + o);
        xi[0] = xv.x;
        xi[1] = xv.y;
        const Bilin<T> bl(xcol, y, xv.x, xv.y, inv_dx, N);
        T c[4];
        ld_quad(phys + 4 * (long long)bl.o00, c);
#pragma unroll
        for (int q = 0; q < 4; ++q) f[q] = mul_rn(bl.w00, c[q]);
        ld_quad(phys + 4 * (long long)bl.o01, c);
#pragma unroll
        for (int q = 0; q < 4; ++q) f[q] = fma(bl.w01, c[q], f[q]);
        ld_quad(phys + 4 * (long long)bl.o10, c);
#pragma unroll
        for (int q = 0; q < 4; ++q) f[q] = fma(bl.w10, c[q], f[q]);
        ld_quad(phys + 4 * (long long)bl.o11, c);
#pragma unroll
        for (int q = 0; q < 4; ++q) f[q] = fma(bl.w11, c[q], f[q]);
        T* dst = S + 2 * xcol + rr;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          dst[q * 2 * N] = b[q];
          dst[(6 + q) * 2 * N] = f[q];
        }
        dst[4 * 2 * N] = xi[0];
        dst[5 * 2 * N] = xi[1];
        if (L.has_q)
          dst[10 * 2 * N] = fma(bl.w11, gld(Q + bl.o11), fma(bl.w10, gld(Q + bl.o10),
                                fma(bl.w01, gld(Q + bl.o01), mul_rn(bl.w00, gld(Q + bl.o00)))));
      }
      __syncthreads();
    }

    // a group's transforms, one loop iteration each: the base fields of the
    // pair (fused; group wg takes fields wg, wg + W, ...), then for each
    // of its products the inverse transforms of two gradients (advection and
    // Strategy-2 products) and the forward transform of the product.  A team
    // shares its one product: set 0 takes d_x and the forward transform, set 1 d_y,
    // and, Strategy 2, sets 2 and 3 the values at x + xi of the two rows; set 0
    // gets theirs through the exchange buffers of sets 2 and 3.
    const bool shared = team && product_heavy(L.pk[p0]);
    cplx<T>* const XY = buf0 + (size_t)(2 - wg) * B * 2 * rs + j;  // set 1's transform
    cplx<T>* const XA = buf0 + (size_t)(3 - wg) * B * 2 * rs + j;  // values at x + xi
    int f = fused ? wg : 4;       // next base field
    int p = shared ? p0 : p0 + wg, sub = shared ? wg : 0;  // next product and its part
    bool basing = true;
    while (true) {
      if (basing && f >= 4) {
        if (fused) __syncthreads();  // base fields complete
        basing = false;
      }
      if (!basing && p >= p1) break;
      const int kind = L.pk[min(p, p1 - 1)], pc = L.pc[min(p, p1 - 1)];
      const bool heavy = product_heavy(kind);
      if (shared && !basing && sub >= 2 && wg >= 2) {
        if (kind == PK_GBAR || (kind == PK_XI && !kin)) {
          const int rr = wg - 2;
          const T* gp = phys + (long long)pc * g.np;
          const T* xp = phys + (long long)PH_XX * g.np + rowoff + rr * N;
          T* dst = reinterpret_cast<T*>(XA) + rr;
#pragma unroll
          for (int m = 0; m < 8; ++m)
            dst[2 * m * G] = bilinear<T>(gp, m * G + j, 2 * yp + rr, gld(xp + m * G), gld(xp + g.np + m * G), inv_dx, N);
        }
        __syncthreads();
        break;
      }
      const bool inv = basing || (heavy && sub < 2);
      if (inv) {
        if (basing && !(d.umask[pg] >> f & 1)) {
          f += W;
          continue;
        }
        const int src = basing ? (f == 0 ? L.i_u : (f == 1 ? L.i_v : (f == 2 ? L.i_h : L.i_z)))
                               : (sub == 0 ? L.pa[p] : L.pb[p]);
        load_rows_ct<T, L_>(x, mix + (long long)src * g.mi, j, g.K);
        if (!basing && sub == 0 && kind != PK_ADV && !shared) {
          // Strategy 2: the values at x + xi (Eqs. xi_evol, barf_xi), by
          // bilinear interpolation, while the gradient rows arrive
          const bool cst = kind == PK_XI && kin;
          const T cv = pc == 0 ? adv_x : adv_y;
          const T* gp = phys + (long long)pc * g.np;
#pragma unroll
          for (int m = 0; m < 8; ++m) {
            acc[m] = mk<T>(cv, cv);
            if (!cst && gath) {
              acc[m] = U[(6 + pc) * N + m * G];
            } else if (!cst) {
              const cplx<T> xx = base(PH_XX, m), xy = base(PH_XY, m);
              const int e = m * G + j;
              acc[m] = mk<T>(bilinear<T>(gp, e, 2 * yp, xx.x, xy.x, inv_dx, N),
                             bilinear<T>(gp, e, 2 * yp + 1, xx.y, xy.y, inv_dx, N));
            }
          }
        }
      } else if (heavy) {
#pragma unroll
        for (int m = 0; m < 8; ++m) x[m] = acc[m];
      } else {
        // products of the base fields alone
        const int fa = kind == PK_ZV || kind == PK_ZU || kind == PK_Q ? PH_Z : (kind == PK_HU || kind == PK_HV ? PH_H : PH_U);
        const int fb = kind == PK_ZU || kind == PK_HU ? PH_U : (kind == PK_Q ? PH_H : PH_V);
        const bool ke = kind == PK_KE, hu = kind == PK_HU || kind == PK_HV;
#pragma unroll
        for (int m = 0; m < 8; ++m) {
          const cplx<T> a = base(fa, m), b = base(fb, m);
          if (ke) x[m] = mk<T>((T)0.5 * (a.x * a.x + b.x * b.x), (T)0.5 * (a.y * a.y + b.y * b.y));
          else if (hu) x[m] = mk<T>(b.x + a.x * b.x, b.y + a.y * b.y);  // depth h = 1 + eta
          else x[m] = mk<T>(a.x * b.x, a.y * b.y);
        }
        if (kind == PK_Q) {
#pragma unroll
          for (int m = 0; m < 8; ++m) {
            const cplx<T> z = base(PH_Z, m), h = base(PH_H, m);
            x[m] = mk<T>((f0 + z.x) / ((T)1 + h.x), (f0 + z.y) / ((T)1 + h.y));
          }
        }
      }
      gfft<T, -1, L_, SYNC>(x, buf0, buf1, w, j, gi, d.tw, gr, inv ? 0 : -L_ - 1);
      if (basing) {
#pragma unroll
        for (int m = 0; m < 8; ++m) U[f * N + m * G] = mk<T>(x[m].y, x[m].x);
        f += W;
      } else if (!inv) {
        store_rows_ct<T, L_, SYNC>(x, buf0, buf1, w, d.pmix + (long long)p * g.mi + (long long)yp * 2 * g.KXP, j, gi,
                                   g.K);
        p += W;
        sub = 0;
      } else {
        if (shared) {
          if (wg == 1) {
#pragma unroll
            for (int m = 0; m < 8; ++m) XY[m * G] = x[m];
          }
          __syncthreads();
          if (wg == 1) break;
          if (kind != PK_ADV) {
            const T cv = pc == 0 ? adv_x : adv_y;
#pragma unroll
            for (int m = 0; m < 8; ++m) acc[m] = kind == PK_XI && kin ? mk<T>(cv, cv) : XA[m * G];
          }
        }
        const int from = sub;
        sub = shared ? 2 : sub + 1;
#pragma unroll 1
        for (int part = from; part < sub; ++part) {
          const bool second = part == 1;
          if (shared && second) {
#pragma unroll
            for (int m = 0; m < 8; ++m) x[m] = XY[m * G];
          }
          if (kind == PK_ADV) {
            // u.grad G (Eq. gtilde-evol) or u.grad D
            const T av = second ? adv_y : adv_x;
#pragma unroll
            for (int m = 0; m < 8; ++m) {
              const cplx<T> ua = kin ? mk<T>(av, av) : base(second ? PH_V : PH_U, m);
              const cplx<T> a = second ? acc[m] : mk<T>(0, 0);
              acc[m] = mk<T>(fma(ua.x, x[m].y, a.x), fma(ua.y, x[m].x, a.y));
            }
          } else {
            // Strategy 2, Eqs. (xi_evol), (barf_xi): w = xi/s, limit u/2 at s = 0
            const bool sz = s0 && !(xf && kind == PK_GBAR);
            const T is = kind == PK_GBAR ? inv_sg : inv_s;
            const T av = second ? adv_y : adv_x;
            const int comp = second ? 1 : 0;
#pragma unroll
            for (int m = 0; m < 8; ++m) {
              cplx<T> wv;
              if (sz) {
                const cplx<T> ua = kin ? mk<T>(av, av) : base(PH_U + comp, m);
                wv = mk<T>((T)0.5 * ua.x, (T)0.5 * ua.y);
              } else {
                const cplx<T> xi = base(PH_XX + comp, m);
                wv = mk<T>(xi.x * is, xi.y * is);
              }
              cplx<T> a = acc[m];
              a.x -= wv.x * x[m].y;
              a.y -= wv.y * x[m].x;
              if (kind == PK_XI && pc == comp) {
                a.x -= wv.x;
                a.y -= wv.y;
              }
              acc[m] = a;
            }
          }
        }
      }
    }
  };
  if constexpr (WARP) dispatch_L<4, 8>(d.g.log2N, body);
  else dispatch_L<4, 11>(d.g.log2N, body);
}

// ---------------------------------------------------------------------------
// a4 and the next stage's a1 in one kernel: forward y-FFT and 2/3 mask of the
// products, right-hand sides, the stepper's combination with the integrating
// factor, and the inverse y-FFTs of the new stage values.  Everything between
// the two transforms is pointwise in (ky, kx), and a forward transform leaves
// position k of a column with the thread that feeds position k to an inverse
// one, so the new value of a field goes from the product's transform to its
// derivatives' transforms through registers.
//
// Separate kernels (forward pass, update, inverse pass) moved 96 spectral and
// 27 mixed fields per stage of a Strategy-1 run with four means (products and
// stage values written and read back, each once per reader); this one moves
// 45 and 27, in one launch instead of three.
//
// Local block = (task, kx tile of C = 2^lC columns); thread t works on column
// c = t mod C and rows n = j + m N/8 (j = t div C, m < 8).  A warp's accesses
// to the spectral fields are contiguous (tile-blocked layout), those to the
// mixed fields runs of C columns x 2 rows.  (With both layouts [row][kx], runs
// of C columns, the kernel was bound by the number of 32-byte requests: 309 us
// at 2048^2 with 4 columns, 608 us with 2.)  A task owns one or two evolved fields: CT_UV (u and v, with
// the products zeta v, zeta u, |u|^2/2; their mixed fields and zeta's), CT_H,
// CT_E2 (the two-dimensional Euler vorticity and its slaved velocity), CT_KIN
// (the kinematic model's u, v, h), CT_G (a mean field and its Eulerian
// accumulator), CT_P (a displacement component).  Only u, v and h are read by
// other tasks (linear terms, f_hat), so only their stage values go to memory;
// they alternate between two buffers, because the other tasks of the launch
// read the previous ones.  stage = -1 only transforms: the mixed fields of the
// state y, before the first step of a replay; with STAGE_FINAL set the mixed
// fields are left out, after its last.
//   RK4   stage 0: a = N(y_n)      acc = E^2 a            y1 = E (y_n + dt/2 a)
//         stage 1: b = N(y1)       acc += 2 E b           y2 = E y_n + dt/2 b
//         stage 2: c = N(y2)       acc += 2 E c           y3 = E^2 y_n + dt E c
//         stage 3: d = N(y3)       y_{n+1} = E^2 y_n + dt/6 (acc + d)
//   Heun  stage 0: acc = E^2 a, y1 = E^2 (y_n + dt a);  stage 1: y_{n+1} =
//         E^2 y_n + dt/2 (acc + b)
//   Euler stage 0: acc = dt E^2 a;  stage 1 (no products): y_{n+1} = E^2 y_n
//         + acc (two launches: the first reads other fields' y_n)
// with E = exp(-nu |k|^2p dt/2).
// The code is kept small (one transform instance for both directions, the
// inverse as a forward transform of swapped parts; the update in a rolled
// loop): a block runs each instruction only a few times, and with the
// transforms and updates of every task unrolled the kernel waited for
// instruction fetches (2048^2: 528 us).
// Smem: C exchange-buffer pairs (col_buf_stride) per part, then 6 complex per
// thread of a part (its parked values: the positions m = 3, 4 of a column, n in
// [3N/8, 5N/8), lie outside the 2/3 box).
__device__ __forceinline__ float kahan_add_rn(float sum, float add, float& comp) {
  const float yk = __fsub_rn(add, comp);
  const float t = __fadd_rn(sum, yk);
  comp = __fsub_rn(__fsub_rn(t, sum), yk);
  return t;
}
__device__ __forceinline__ double kahan_add_rn(double sum, double add, double& comp) {
  const double yk = __dsub_rn(add, comp);
  const double t = __dadd_rn(sum, yk);
  comp = __dsub_rn(__dsub_rn(t, sum), yk);
  return t;
}

// Two-dimensional Euler model: the velocity of the vorticity zeta at mode m of
// buffer b, through the streamfunction (lap psi = zeta, u = -d_y psi,
// v = d_x psi): u_hat = i ky zeta_hat/|k|^2, v_hat = -i kx zeta_hat/|k|^2, zero
// at k = 0; written beside zeta.
template <typename T>
__device__ __forceinline__ void slave_velocity(cplx<T>* b, const Layout& L, int ms, int m, T kxf, T kyf, cplx<T> z) {
  const T k2 = kxf * kxf + kyf * kyf;
  const T inv = k2 > (T)0 ? (T)1 / k2 : (T)0;
  gst(b + L.f_u * ms + m, mk<T>(-kyf * z.y * inv, kyf * z.x * inv));
  gst(b + L.f_v * ms + m, mk<T>(kxf * z.y * inv, -kxf * z.x * inv));
}

// y_{n+1} = E^2 y_n + inc, with the factor E^2 given as the unevaluated sum
// e2h + e2l (the part e2l y_n joins the increment); compensated if `kahan`
// (cc: the compensation term, replaced).
template <typename T>
__device__ __forceinline__ cplx<T> commit_mode(bool kahan, T e2h, T e2l, cplx<T> yn, cplx<T>& cc, cplx<T> inc) {
  inc.x = fma(yn.x, e2l, inc.x);
  inc.y = fma(yn.y, e2l, inc.y);
  if (kahan) {
    cc.x *= e2h;
    cc.y *= e2h;
    return mk<T>(kahan_add_rn(yn.x * e2h, inc.x, cc.x), kahan_add_rn(yn.y * e2h, inc.y, cc.y));
  }
  return mk<T>(fma(yn.x, e2h, inc.x), fma(yn.y, e2h, inc.y));
}

// v or -v, by an integer instruction in FP64.
__device__ __forceinline__ float neg_if(bool n, float v) { return n ? -v : v; }
__device__ __forceinline__ double neg_if(bool n, double v) {
  return __hiloint2double(__double2hiint(v) ^ (n ? (int)0x80000000 : 0), __double2loint(v));
}

// Integer as a T; FP64 by integer instructions (a conversion is an FP64-pipe
// instruction), |k| < 2^20.
__device__ __forceinline__ float to_real(int k, float) { return (float)k; }
__device__ __forceinline__ double to_real(int k, double) {
  const unsigned a = (unsigned)abs(k);
  const int lz = __clz((int)a);
  const unsigned hi = ((a << lz) >> 11) + ((unsigned)(1022 + 31 - lz) << 20);
  return __hiloint2double(a ? (int)(hi | ((unsigned)k & 0x80000000u)) : 0, 0);
}

// The run's last block to finish its step advances the step counter (every block
// of the run has read it before taking its ticket).
template <typename T> __device__ __forceinline__ void finish_step(const RunDesc<T>& d, int kt) {
  __syncthreads();
  if (threadIdx.x == 0) {
    const long long n = *d.ctr;
    __threadfence();
    const unsigned t = atomicAdd(d.ticket, 1u);
    if (t == (unsigned)d.nb[kt] - 1u) {
      // (visible to the next kernels: they wait for the end of this one)
      *d.ticket = 0u;
      *d.ctr = n + 1;
    }
  }
}

template <typename T> __device__ __forceinline__ cplx<T> cswap(cplx<T> a) { return mk<T>(a.y, a.x); }

// Column-stage kernels by the largest block: FP64 128 threads (grids up to
// 512^2: few warps per SM, so many registers and three modes in flight, which spill 250
// to 410 bytes at 255 registers; two spill none: a Strategy-1 step 143.1 against 141.9 us
// at 64^2, but 295.7 against 300.5 at 256^2 and 610 against 647 at 512^2) and 256;
// FP32 256 (to 512^2), 512 (1024^2) and 1024 (2048^2).
// PARTS: a task's steps are shared out over two or four parts of a block, each
// with its own exchange buffers and barrier (block barriers where a value passes
// between them): while a launch has about one block per SM its time is the
// longest task's chain, which halves cut from 6 transforms and 2 updates to 3
// and 1 (CT_UV) and from 3 and 1 to 2 and 1 (CT_G), and quarters (N <= 128) to 2 and 1 for
// every task.  Step of one Strategy-1 run, whole blocks -> halves: 64^2 FP64 0.240 ->
// 0.188 ms, 256^2 FP32 0.078 -> 0.071 ms; at 512^2, more than a block per SM, no
// difference; quarters: see QUAD_BLOCKS.  (Quarters at 256^2 in FP32, 512 threads
// and one block per SM, lose: the kernel alone 8.1 -> 9.6 us.)
constexpr int STAGE_FINAL = 256;
template <typename T, int MAXT, int PARTS> struct ColShape {
  static constexpr bool f32 = sizeof(T) == 4;
  static constexpr int LO = f32 ? (MAXT <= 256 ? 4 : (MAXT <= 512 ? 10 : 11)) : (MAXT <= 128 ? 4 : 10);
  static constexpr int HI = PARTS == 4 ? 7 : PARTS == 2 ? 8 : f32 ? (MAXT <= 256 ? 9 : LO) : (MAXT <= 128 ? 9 : 11);
  static constexpr int NB = f32 ? 2 : (MAXT <= 128 ? 3 : 1);  // modes whose loads are issued together
  static constexpr int BLOCKS = MAXT <= 512 ? 2 : 1;
};
template <typename T, int MAXT, int PARTS>
__global__ void __launch_bounds__(MAXT, ColShape<T, MAXT, PARTS>::BLOCKS) k_stage_col(const RunDesc<T>* __restrict__ runs,
                                                                              const int* __restrict__ start,
                                                                              int nruns, int stage_arg) {
  const bool final_step = stage_arg >= 0 && (stage_arg & STAGE_FINAL);
  const int stage = stage_arg < 0 ? stage_arg : stage_arg & ~STAGE_FINAL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned red[GRedWords<T>::value];  // FP64 transforms
  const int r = find_run(start, nruns, blockIdx.x);
  LM_STAGE_DESC(T);  // field and product lookups from shared memory
  pdl_wait();  // state written by the previous kernels: only after this
  pdl_release();
  const int lb = blockIdx.x - start[r];
  dispatch_L<ColShape<T, MAXT, PARTS>::LO, ColShape<T, MAXT, PARTS>::HI>(d.g.log2N, [&](auto Lc) {
    constexpr int L = decltype(Lc)::value, N = 1 << L, G = N / 8;
    constexpr int NB = ColShape<T, MAXT, PARTS>::NB;
    const Layout& Y = d.L;
    const int K = d.g.K, KXP = d.g.KXP, ms = (int)d.g.ms;
    const int lC = d.lC, C = 1 << lC;
    const int ntile = KXP >> lC;
    const int task = lb / ntile, tile = lb - task * ntile;
    const ColTask& ct = Y.ct[task];
    const int kind = ct.kind, slot = ct.slot;
    constexpr int SYNC = PARTS == 4 ? 4 : PARTS == 2 ? 3 : 2;
    const int ps = blockDim.x / PARTS;  // threads per part
    const int part = PARTS > 1 ? threadIdx.x / ps : 0, tid = threadIdx.x - part * ps;
    const int c = tid & (C - 1), j = tid >> lC;
    const int st = d.c.stepper;
    const bool begin = stage < 0;
    const bool last = stage == stage_count(st) - 1;  // commits y_{n+1}
    const bool euler0 = st == 2 && stage == 0;       // forward Euler's first pass
    const bool commit = st == 2 && stage == 1;       // and its second: no products
    const long long nstep = *d.ctr;
    auto sd = [&]() { return stage_time<T>(nstep, stage, d.cdt, st); };
    const int kx = (tile << lC) + c;
    const T kxf = to_real(kx, (T)0);
    const bool col = kx <= K;
    const bool e2 = Y.model == 2, kin = Y.model == 1;
    const int xs = C * col_buf_stride<T>(N, C);  // exchange buffers of a part
    cplx<T>* b0 = reinterpret_cast<cplx<T>*>(smem_raw) + part * xs + c * col_buf_stride<T>(N, C);
    cplx<T>* park = reinterpret_cast<cplx<T>*>(smem_raw) + PARTS * xs + tid;
    const GRed gr = {red + part * (GRED_WORDS / 2 / PARTS), lC, tid, ps};
    int w = 0;
    cplx<T> x[8];
    // the column's first mode, the row stride of its modes, and its elements
    // of a mixed field (row n = j + m G at mx + m * mG)
    constexpr int CS = spec_tile<T>();
    const int m00 = (kx / CS) * (d.g.NY * CS) + kx % CS;
    const int mx = (j >> 1) * 2 * KXP + 2 * kx + (j & 1), mG = G * KXP;
    // wavenumber of the thread's position s = 0..5 (m = s or s + 2), and
    // whether it lies in the box
    auto kyof = [&](int s) { return j + s * G - (s >= 3 ? 6 * G : 0); };
    auto inband = [&](int s) { return col && kyof(s) <= K && kyof(s) >= -K; };
    const cplx<T>* yin = stage_input(d, stage);
    cplx<T>* yout = last || begin ? d.y : (stage == 1 ? d.ysb : d.ysa);
    auto store_park = [&]() {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        park[i * ps] = x[i];
        park[(3 + i) * ps] = x[5 + i];
      }
    };

    // The task's update of field f (and, fe >= 0, of the Eulerian accumulator
    // fe) at the thread's modes: x, the transformed product (times 1/N), is
    // replaced by the new values.  fa, fb: stage inputs read with it (-1:
    // none).  Loads are unconditional over the thread's positions, from
    // clamped addresses (a load under a per-lane condition waits where the
    // lanes rejoin), and issued together for NB modes.  Before the commit the
    // combinations of all steppers and stages are acc' = [acc +] cr rhs,
    // y' = ca y_n + cb rhs.
    auto update = [&](int f, int fe, int fa, int fb) {
      const int role = Y.frole[f];
      const int cls = Y.fclass[f];
      const bool damped = cls != IF_NONE;
      const T* ef = d.ef + (damped ? 3 * cls * ms : 0);
      // xi-first scheme (Strategy 2, forward Euler): xi steps by 2 dt on even
      // steps, gbar on odd ones (integrating factor over 2 dt: E^4)
      const bool x1 = Y.scheme == SCHEME_XI_FIRST && (role == R_P || role == R_G);
      const bool act = !x1 || ((role == R_P) == ((nstep & 1) == 0));
      const bool add = st == 0 && stage > 0;
      const bool kah = sizeof(T) == 4 && d.comp && Y.fkahan[f];  // (FP64 runs have no compensation)
      const bool keep = role <= R_H && !euler0;  // stage values that other tasks read
      cplx<T>* const yf = d.y + f * ms;
      cplx<T>* const af = d.acc + f * ms;
      cplx<T>* const ye = d.y + max(fe, 0) * ms;
      cplx<T>* const ae = d.acc + max(fe, 0) * ms;
      const cplx<T>* const qa = yin + max(fa, 0) * ms;
      const cplx<T>* const qb = yin + max(fb, 0) * ms;
      const T dt = d.cdt;
      const cplx<T> z = mk<T>(0, 0);
      // right-hand sides rr of the NB modes from s0 on (wavenumbers ky) from
      // the transformed products tv and the stage inputs pa, pb; fh: the
      // averaged scalar's f_hat (CT_G).  Branches are taken once for the NB
      // modes, whose arithmetic then overlaps.
      auto rhs = [&](int s0, const T* ky, const cplx<T>* tv, const cplx<T>* pa, const cplx<T>* pb, cplx<T>* rr,
                     cplx<T>* fh) {
        if (kind == CT_G) {
          // S1: f - u.grad g (Eq. gtilde-evol), S2: f(x+xi) - w.grad g
          const bool s1 = Y.strategy == 1;
          if (fb >= 0) {
#pragma unroll
            for (int i = 0; i < NB; ++i) fh[i] = csub<T>(cik<T>(pa[i], kxf), cik<T>(pb[i], ky[i]));
          } else {
            const bool pk = fa < 0;
#pragma unroll
            for (int i = 0; i < NB; ++i) fh[i] = pk ? park[(s0 + i) * ps] : pa[i];
          }
#pragma unroll
          for (int i = 0; i < NB; ++i) rr[i] = s1 ? csub<T>(fh[i], tv[i]) : tv[i];
        } else if (kind == CT_P) {
          // S1: d_t D = s u - u.grad D; S2: the product holds u(x+xi) - w - w.grad xi
          const bool s1 = Y.strategy == 1;
          const T sv = sd(), av = slot == 0 ? d.cadvx : d.cadvy;
#pragma unroll
          for (int i = 0; i < NB; ++i) {
            const cplx<T> u = kin ? mk<T>(kx == 0 && kyof(s0 + i) == 0 ? av : (T)0, 0) : pa[i];
            rr[i] = s1 ? csub<T>(cscale<T>(u, sv), tv[i]) : tv[i];
          }
        } else if (kind == CT_UV) {
          // shallow-water momentum, Eq. (sw_eqs_dimless); pa: h, pb: v or u,
          // parked |u|^2/2: u_t = f0 v + (zeta v) - d_x B, v_t = -(f0 u + (zeta u)) - d_y B
          const bool iu = role == R_U;
          const T sg = iu ? (T)1 : (T)-1, f0 = d.cf0, c2 = d.cc2;
#pragma unroll
          for (int i = 0; i < NB; ++i) {
            const cplx<T> pk = park[(s0 + i) * ps];
            const cplx<T> Bq = mk<T>(fma(pa[i].x, c2, pk.x), fma(pa[i].y, c2, pk.y));
            const cplx<T> lin = mk<T>(fma(pb[i].x, f0, tv[i].x), fma(pb[i].y, f0, tv[i].y));
            const T k = iu ? kxf : ky[i];
            // (FP64: the sign by an integer instruction)
            const T lx = sizeof(T) == 8 ? neg_if(!iu, lin.x) : sg * lin.x, ly = sizeof(T) == 8 ? neg_if(!iu, lin.y) : sg * lin.y;
            rr[i] = mk<T>(fma(Bq.y, k, lx), fma(Bq.x, -k, ly));
          }
        } else if (kind == CT_KIN) {
#pragma unroll
          for (int i = 0; i < NB; ++i) rr[i] = cik<T>(pa[i], -(kxf * d.cadvx + ky[i] * d.cadvy));
        } else {
          // -div(h u), or the two-dimensional Euler vorticity's -div(u zeta);
          // the x component parked
#pragma unroll
          for (int i = 0; i < NB; ++i)
            rr[i] = csub<T>(z, cadd<T>(cik<T>(park[(s0 + i) * ps], kxf), cik<T>(tv[i], ky[i])));
        }
      };
      // NB modes at a time; t rotates
      cplx<T> t[6] = {x[0], x[1], x[2], x[5], x[6], x[7]};
      if (!last) {
#pragma unroll 1
        for (int s0 = 0; s0 < 6; s0 += NB) {
          cplx<T> yn[NB], ac[NB], pa[NB], pb[NB], ea[NB], nv[NB];
          T E[NB];
          int ml[NB];
#pragma unroll
          for (int i = 0; i < NB; ++i) {
            ml[i] = (min(max(kyof(s0 + i), -K), K) + K) * CS + m00;
            yn[i] = yf[ml[i]];
            ac[i] = pa[i] = pb[i] = ea[i] = z;
            E[i] = (T)1;
          }
          if (damped) {
#pragma unroll
            for (int i = 0; i < NB; ++i) E[i] = ef[ml[i]];
          }
          if (fa >= 0) {
#pragma unroll
            for (int i = 0; i < NB; ++i) pa[i] = qa[ml[i]];
          }
          if (fb >= 0) {
#pragma unroll
            for (int i = 0; i < NB; ++i) pb[i] = qb[ml[i]];
          }
          if (add) {
#pragma unroll
            for (int i = 0; i < NB; ++i) ac[i] = af[ml[i]];
            if (fe >= 0) {
#pragma unroll
              for (int i = 0; i < NB; ++i) ea[i] = ae[ml[i]];
            }
          }
          T ky[NB];
          bool in[NB];
          cplx<T> rr[NB], fh[NB];
#pragma unroll
          for (int i = 0; i < NB; ++i) {
            ky[i] = to_real(kyof(s0 + i), (T)0);
            in[i] = inband(s0 + i);
            fh[i] = z;
          }
          rhs(s0, ky, t, pa, pb, rr, fh);
          // coefficients: RK4, Heun (E^2, E^2, dt E^2) and forward Euler (acc
          // alone, dt E^2; xi-first means 2 dt E^4)
          const T hdt = (T)0.5 * dt;
#pragma unroll
          for (int i = 0; i < NB; ++i) {
            const T e1 = E[i], ee = e1 * e1;
            T cr = stage == 0 ? ee : (T)2 * e1;
            T ca = stage == 2 ? ee : e1;
            T cb;
            if (sizeof(T) == 8) {
              // few FP64 operations: both sides of a choice between products are
              // evaluated, so the choice is between their factors
              cb = (st == 0 && stage < 2 ? hdt : dt) * (st != 0 ? ee : (stage == 1 ? (T)1 : e1));
              if (st != 0) ca = ee;
              if (st == 2) {
                asm volatile("");  // a branch
                cr = x1 ? (T)2 * dt * ee * ee : dt * ee;
              }
            } else {
              cb = stage == 0 ? hdt * e1 : (stage == 1 ? hdt : dt * e1);
              if (st != 0) {
                cr = ca = ee;
                cb = dt * ee;
                if (st == 2) cr = x1 ? (T)2 * dt * ee * ee : dt * ee;
              }
            }
            nv[i] = z;
            if (sizeof(T) == 4 || st != 2) {  // (forward Euler's first pass has no stage value)
              if (sizeof(T) == 8) asm volatile("");
              nv[i] = mk<T>(fma(ca, yn[i].x, cb * rr[i].x), fma(ca, yn[i].y, cb * rr[i].y));
            }
            ac[i] = mk<T>(fma(cr, rr[i].x, ac[i].x), fma(cr, rr[i].y, ac[i].y));
            if (in[i] && act) gst(af + ml[i], ac[i]);
            nv[i] = in[i] ? nv[i] : z;
          }
          if (fe >= 0) {
            // Eq. (ave), undamped
            const T ce = st == 0 ? (stage == 0 ? (T)1 : (T)2) : (st == 1 ? (T)1 : dt);
#pragma unroll
            for (int i = 0; i < NB; ++i)
              if (in[i]) gst(ae + ml[i], mk<T>(fma(ce, fh[i].x, ea[i].x), fma(ce, fh[i].y, ea[i].y)));
          }
          if (keep) {
#pragma unroll
            for (int i = 0; i < NB; ++i)
              if (in[i]) gst(yout + f * ms + ml[i], nv[i]);
            if (kind == CT_E2) {
#pragma unroll
              for (int i = 0; i < NB; ++i)
                if (in[i]) slave_velocity<T>(yout, Y, ms, ml[i], kxf, ky[i], nv[i]);
            }
          }
#pragma unroll
          for (int i = 0; i < 6; ++i) t[i] = i < 6 - NB ? t[(i + NB) % 6] : nv[i < 6 - NB ? 0 : i - (6 - NB)];
        }
      } else {
        // final stage: y_{n+1} = E^2 y_n + inc, with inc = dt/6 (acc + d) (RK4),
        // dt/2 (acc + b) (Heun) or forward Euler's increment acc
        const T ci = sizeof(T) == 8 ? d.cci : (st == 0 ? dt / (T)6 : (st == 1 ? dt / (T)2 : (T)1));
#pragma unroll 1
        for (int s0 = 0; s0 < 6; s0 += NB) {
          cplx<T> yn[NB], ac[NB], cc[NB], pa[NB], pb[NB], en[NB], ea[NB], ec[NB], nv[NB];
          T eh[NB], el[NB];
          int ml[NB];
#pragma unroll
          for (int i = 0; i < NB; ++i) {
            ml[i] = (min(max(kyof(s0 + i), -K), K) + K) * CS + m00;
            yn[i] = yf[ml[i]];
            ac[i] = af[ml[i]];
            cc[i] = pa[i] = pb[i] = en[i] = ea[i] = ec[i] = z;
            eh[i] = (T)1;
            el[i] = (T)0;
          }
          if (damped) {
#pragma unroll
            for (int i = 0; i < NB; ++i) {
              eh[i] = ef[ms + ml[i]];
              el[i] = ef[2 * ms + ml[i]];
            }
          }
          if (fa >= 0) {
#pragma unroll
            for (int i = 0; i < NB; ++i) pa[i] = qa[ml[i]];
          }
          if (fb >= 0) {
#pragma unroll
            for (int i = 0; i < NB; ++i) pb[i] = qb[ml[i]];
          }
          if (kah) {
#pragma unroll
            for (int i = 0; i < NB; ++i) cc[i] = d.comp[f * ms + ml[i]];
          }
          if (fe >= 0) {
#pragma unroll
            for (int i = 0; i < NB; ++i) {
              en[i] = ye[ml[i]];
              ea[i] = ae[ml[i]];
            }
            if (sizeof(T) == 4 && d.comp) {
#pragma unroll
              for (int i = 0; i < NB; ++i) ec[i] = d.comp[fe * ms + ml[i]];
            }
          }
          T ky[NB];
          bool in[NB];
          cplx<T> rr[NB], fh[NB];
#pragma unroll
          for (int i = 0; i < NB; ++i) {
            ky[i] = to_real(kyof(s0 + i), (T)0);
            in[i] = inband(s0 + i);
            rr[i] = fh[i] = z;
          }
          if (!commit) rhs(s0, ky, t, pa, pb, rr, fh);
          if (x1) {
            if (sizeof(T) == 8) asm volatile("");  // a branch
            // E^4 = (eh + el)^2 to the same precision (exact product of eh by fma)
#pragma unroll
            for (int i = 0; i < NB; ++i) {
              const T h2 = eh[i] * eh[i];
              el[i] = fma(eh[i], eh[i], -h2) + (T)2 * eh[i] * el[i];
              eh[i] = h2;
            }
          }
          cplx<T>* const cf = d.comp + f * ms;
#pragma unroll
          for (int i = 0; i < NB; ++i) {
            cplx<T> inc = ac[i];
            if (sizeof(T) == 4 || !commit) {  // (forward Euler commits acc itself)
              if (sizeof(T) == 8) asm volatile("");
              inc = cscale<T>(cadd<T>(ac[i], rr[i]), ci);
            }
            nv[i] = commit_mode<T>(kah, eh[i], el[i], yn[i], cc[i], inc);
            if (!act) nv[i] = yn[i];
            if (in[i] && act) {
              gst(yf + ml[i], nv[i]);
              if (kah) gst(cf + ml[i], cc[i]);
            }
            nv[i] = in[i] ? nv[i] : z;
          }
          if (fe >= 0) {
            const bool ke = sizeof(T) == 4 && d.comp != nullptr;
            cplx<T>* const cfe = d.comp + fe * ms;
#pragma unroll
            for (int i = 0; i < NB; ++i) {
              const cplx<T> v = commit_mode<T>(ke, (T)1, (T)0, en[i], ec[i], cscale<T>(cadd<T>(ea[i], fh[i]), ci));
              if (in[i]) {
                gst(ye + ml[i], v);
                if (ke) gst(cfe + ml[i], ec[i]);
              }
            }
          }
          if (kind == CT_E2) {
#pragma unroll
            for (int i = 0; i < NB; ++i)
              if (in[i]) slave_velocity<T>(yout, Y, ms, ml[i], kxf, ky[i], nv[i]);
          }
#pragma unroll
          for (int i = 0; i < 6; ++i) t[i] = i < 6 - NB ? t[(i + NB) % 6] : nv[i < 6 - NB ? 0 : i - (6 - NB)];
        }
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        x[i] = t[i];
        x[5 + i] = t[3 + i];
      }
    };
    auto load_park = [&]() {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        x[i] = park[i * ps];
        x[5 + i] = park[(3 + i) * ps];
      }
    };
    // field f of the stage's output at the thread's positions (u, v, h only:
    // written by this thread, or the state)
    auto load_out = [&](int f) {
      const cplx<T>* y = yout + f * ms + m00;
#pragma unroll
      for (int s = 0; s < 6; ++s) {
        const cplx<T> v = gld(y + (min(max(kyof(s), -K), K) + K) * CS);
        x[s < 3 ? s : s + 2] = inband(s) ? v : mk<T>(0, 0);
      }
    };

    // The task's steps: transforms of its products (a forward transform and
    // what becomes of it) and of its mixed fields IFFT_y(op(value)), op in
    // {id, d_x, d_y, curl}, as a forward transform of swapped parts.  None of
    // the latter after forward Euler's first pass, or a replay's last step;
    // only these when beginning.
    const bool outs = !euler0 && !final_step;
    for (int q = 0; q < ct.n; ++q) {
      const int p = ct.prod[q], act = ct.act[q], op = ct.op[q];
      const bool fwd = op < 0;
      if (PARTS > 1 && ct.bar[q]) __syncthreads();
      if ((fwd ? begin : !outs) || (PARTS > 1 && ct.part[q] != part)) continue;
      if (fwd) {
        if (p >= 0 && !commit) {
          const cplx<T>* src = d.pmix + (long long)p * d.g.mi + mx;
#pragma unroll
          for (int m = 0; m < 8; ++m) x[m] = src[m * mG];
        }
      } else {
        // the value: in x after an update, or the parked one, or (when
        // beginning, and for the fields of CT_UV, CT_E2 and CT_KIN) in memory
        if (begin || act == CA_MEM) {
          if (op == OP_CURL) {
            // i kx v - i ky u
            cplx<T> u[6];
            load_out(Y.f_u);
#pragma unroll
            for (int s = 0; s < 6; ++s) u[s] = x[s < 3 ? s : s + 2];
            load_out(Y.f_v);
#pragma unroll
            for (int s = 0; s < 6; ++s)
              x[s < 3 ? s : s + 2] = csub<T>(cik<T>(x[s < 3 ? s : s + 2], kxf), cik<T>(u[s], to_real(kyof(s), (T)0)));
          } else {
            load_out(ct.fld[q]);
          }
        } else if (act == CA_PARKED) {
          load_park();
        }
#pragma unroll
        for (int s = 0; s < 6; ++s) {
          cplx<T> v = x[s < 3 ? s : s + 2];
          if (op == OP_DX) v = cik<T>(v, kxf);
          else if (op == OP_DY) v = cik<T>(v, to_real(kyof(s), (T)0));
          x[s < 3 ? s : s + 2] = cswap<T>(v);
        }
        x[3] = x[4] = mk<T>(0, 0);
      }
      if (!(fwd && (p < 0 || commit)))
        gfft<T, -1, L, SYNC>(x, b0, b0 + row_stride<T>(N), w, j, part, d.tw, gr, fwd ? -L : 0);
      if (fwd) {
        if (act != CA_PARK && act != CA_KEEP) {
          int fe = -1, fa = -1, fb = -1;
          const int fu = ct.fld[q];
          if (kind == CT_UV) {
            fa = Y.f_h;
            fb = act == CA_U ? Y.f_v : Y.f_u;
          } else if (kind == CT_KIN) {
            fa = fu;
          } else if (kind == CT_P) {
            if (Y.strategy == 1 && !kin) fa = slot == 0 ? Y.f_u : Y.f_v;
          } else if (kind == CT_G) {
            const int sc = Y.lmf[slot];
            fe = Y.f_e[slot];
            if ((Y.strategy == 1 || fe >= 0) && sc != LMF_Q) {
              fa = sc == LMF_ZETA ? (e2 ? Y.f_h : Y.f_v) : (sc == LMF_H ? Y.f_h : (sc == LMF_U ? Y.f_u : Y.f_v));
              if (sc == LMF_ZETA && !e2) fb = Y.f_u;
            }
          }
          update(fu, fe, fa, fb);
        }
        if (act == CA_PARK || act == CA_UPD_PARK) store_park();
      } else {
        cplx<T>* dst = d.mix + (long long)p * d.g.mi + mx;
#pragma unroll
        for (int m = 0; m < 8; ++m) gst(dst + m * mG, cswap<T>(x[m]));
      }
    }
  });
  if (stage == stage_count(d.c.stepper) - 1) finish_step(d, KT_COL_STAGE);
}

// ---------------------------------------------------------------------------
// The kinematic model's u, v and h when nothing is averaged: no products, so no
// transforms, one pointwise pass per stage.  Bound by FP64 issue or memory (large
// grids) or by the launch (small ones): a thread takes the three fields of a mode
// (one wavenumber and one set of coefficients for them, their loads issued
// together), one mode up to 512^2 (short chains, many blocks), two above; no
// shared memory and at most 80 registers.  A step, as blocks of the column stage
// (255 registers in FP64, its exchange buffers allocated) -> this: @@
__host__ __device__ __forceinline__ int kin_modes(int N) { return N >= 1024 ? 512 : 256; }
template <typename T>
__global__ void __launch_bounds__(256, 3) k_stage_kin(const RunDesc<T>* __restrict__ runs,
                                                      const int* __restrict__ start, int nruns, int stage) {
  const int r = find_run(start, nruns, blockIdx.x);
  const RunDesc<T>& d = runs[r];
  const int st = d.c.stepper, ms = (int)d.g.ms, NY = d.g.NY, K = d.g.K, per = kin_modes(d.g.N);
  constexpr int CS = spec_tile<T>();
  const bool last = stage == stage_count(st) - 1;
  const int m0 = (blockIdx.x - start[r]) * per, m1 = min(ms, m0 + per);
  // u and v are of class IF_DYN; h too, or undamped
  const bool hdamped = d.L.fclass[2] != IF_NONE;
  const T* const ef = d.ef;
  const T dt = d.cdt, ax = d.cadvx, ay = d.cadvy;
  const cplx<T>* const yin = stage_input(d, stage);
  cplx<T>* const yout = stage == 1 ? d.ysb : d.ysa;
  cplx<T>* const y = d.y;
  cplx<T>* const acc = d.acc;
  // acc' = [acc +] cr rhs, y' = ca y_n + cb rhs (see k_stage_col)
  struct Coef { T cr, ca, cb; };
  const T hdt = (T)0.5 * dt;
  auto coef = [&](T e1) {
    Coef c;
    if (st != 0) {
      c.cr = c.ca = e1 * e1;
      c.cb = dt * c.ca;
    } else if (stage == 0) {
      c.cr = e1 * e1;
      c.ca = e1;
      c.cb = hdt * e1;
    } else {
      c.cr = (T)2 * e1;
      c.ca = stage == 1 ? e1 : e1 * e1;
      c.cb = stage == 1 ? hdt : dt * e1;
    }
    return c;
  };
  const T ci = d.cci;
  const bool radd = !last || st != 2;              // the stage adds a right-hand side
  const bool racc = last || (st == 0 && stage > 0);  // acc is read
  pdl_wait();  // state written by the previous kernels: only after this
  pdl_release();
  for (int m = m0 + threadIdx.x; m < m1; m += blockDim.x) {
    const int tile = m / (NY * CS), e = m - tile * NY * CS;
    const int kx = tile * CS + e % CS, ky = e / CS - K;
    if (kx > K) continue;
    cplx<T> yn[3], rr[3], ac[3];
    T e1[2] = {(T)1, (T)0};  // E, or E^2 as hi + lo at the commit
    if (last) {
      e1[0] = ef[ms + m];
      e1[1] = ef[2 * ms + m];
    } else {
      e1[0] = ef[m];
    }
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      yn[f] = y[f * ms + m];
      rr[f] = ac[f] = mk<T>(0, 0);
      if (radd) rr[f] = yin[f * ms + m];
      if (racc) ac[f] = acc[f * ms + m];
    }
    const T kc = to_real(kx, (T)0) * ax + to_real(ky, (T)0) * ay;
    if (last) {
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        const bool dm = f < 2 || hdamped;
        const cplx<T> inc = st == 2 ? ac[f] : cscale<T>(cadd<T>(ac[f], cik<T>(rr[f], -kc)), ci);
        cplx<T> cc = mk<T>(0, 0);
        y[f * ms + m] = commit_mode<T>(false, dm ? e1[0] : (T)1, dm ? e1[1] : (T)0, yn[f], cc, inc);
      }
    } else {
      const Coef c0 = coef(e1[0]), ch = hdamped ? c0 : coef((T)1);
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        const Coef c = f < 2 ? c0 : ch;
        const cplx<T> q = cik<T>(rr[f], -kc);
        if (st == 2) {
          acc[f * ms + m] = cscale<T>(q, c.cb);
        } else {
          acc[f * ms + m] = mk<T>(fma(c.cr, q.x, ac[f].x), fma(c.cr, q.y, ac[f].y));
          yout[f * ms + m] = mk<T>(fma(c.ca, yn[f].x, c.cb * q.x), fma(c.ca, yn[f].y, c.cb * q.y));
        }
      }
    }
  }
  if (last) finish_step(d, KT_KIN);
}

}  // namespace lm
