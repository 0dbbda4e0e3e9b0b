// common.cuh -- types, data layout and kernel parameter blocks shared by the
// GB300 kernels of the Lagrangian-mean shallow-water library.
//
// Data layout in HBM (all complex arrays interleaved re/im):
//   spectral field  : tiles of CT = 4 (FP32) or 2 (FP64) consecutive kx, each
//                     [ky_idx][kx mod CT], ky_idx = ky + K in [0, 2K], kx in
//                     [0, KXP) (K = floor((N-1)/3) is the 2/3-rule cutoff; KXP
//                     is K+1 rounded up to a multiple of 4; columns kx > K are
//                     zero): a column tile is one contiguous run
//   column-transformed intermediate ("mixed" field, physical y, spectral kx):
//                     [y/2][kx][y mod 2], kx in [0, KXP)
//   physical field  : [y][x] real, row-major.
// The mixed layout interleaves pairs of rows: the row pass, which transforms
// two rows as one complex sequence, reads and writes both with one 16- or
// 32-byte access per lane, and the column pass moves runs of 2 rows x C
// columns.  (The transforms around the stepping use the same layouts, their
// mixed fields in FP64.)
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace lm {

template <typename T> struct CT;
template <> struct CT<float> { typedef float2 type; };
template <> struct CT<double> { typedef double2 type; };
template <typename T> using cplx = typename CT<T>::type;

template <typename T> __host__ __device__ __forceinline__ cplx<T> mk(T x, T y) {
  cplx<T> r; r.x = x; r.y = y; return r;
}
template <typename T> __device__ __forceinline__ cplx<T> cadd(cplx<T> a, cplx<T> b) { return mk<T>(a.x + b.x, a.y + b.y); }
template <typename T> __device__ __forceinline__ cplx<T> csub(cplx<T> a, cplx<T> b) { return mk<T>(a.x - b.x, a.y - b.y); }
template <typename T> __device__ __forceinline__ cplx<T> cmul(cplx<T> a, cplx<T> b) {
  return mk<T>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a product that is rounded by itself (never contracted into an addition)
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
template <typename T> __device__ __forceinline__ cplx<T> cscale(cplx<T> a, T s) { return mk<T>(a.x * s, a.y * s); }
// multiply by i*k (spectral derivative)
template <typename T> __device__ __forceinline__ cplx<T> cik(cplx<T> a, T k) { return mk<T>(-a.y * k, a.x * k); }

// Shared-memory position of element n of a transform: one spare slot every
// 8 elements.  Shared memory serves 8-byte accesses per half-warp from 16
// slots of 8 bytes (16-byte accesses per quarter-warp from 8 slots); the
// padding spreads the stride-8 writes of the first radix-8 pass over
// distinct slots.  (An XOR swizzle that also keeps the consecutive accesses
// conflict-free halves the shared-memory wavefronts of the FFT kernels but
// costs more index arithmetic than it saves: the kernels are bound by
// latency, not by shared-memory bandwidth.)
template <typename T>
__host__ __device__ __forceinline__ int sidx(int n) {
  return n + (n >> 3);
}
// floor of a double and its integer value modulo 2^32, by integer instructions
// (FP64 ones, conversions included, take 16 clocks of the SM each): exactly
// floor() and its conversion, which are called for |v| >= 2^30, zeros and
// non-finite values.
__device__ __forceinline__ double floor_int(double v, unsigned& k) {
  const int hi = __double2hiint(v), lo = __double2loint(v);
  const int e = ((hi >> 20) & 0x7ff) - 1023;
  if (e >= 30 || ((hi & 0x7fffffff) | lo) == 0) {
    const double f = floor(v);
    k = (unsigned)(long long)f;
    return f;
  }
  int n = 0;      // |v| truncated
  bool rem = true;  // |v| has a fraction
  if (e >= 0) {
    const unsigned m = ((unsigned)hi & 0xfffffu) | 0x100000u;
    const int sh = 52 - e;  // 23 .. 52
    if (sh >= 32) {
      n = (int)(m >> (sh - 32));
      rem = ((m & ((1u << (sh - 32)) - 1u)) | (unsigned)lo) != 0u;
    } else {
      n = (int)((m << (32 - sh)) | ((unsigned)lo >> sh));
      rem = ((unsigned)lo & ((1u << sh) - 1u)) != 0u;
    }
  }
  if (hi < 0) n = -n - (rem ? 1 : 0);
  k = (unsigned)n;
  // n as a double, exact (|n| <= 2^30)
  const unsigned a = (unsigned)abs(n);
  const int lz = __clz((int)a);
  const unsigned long long mant = (unsigned long long)(a << lz) << 21;
  const unsigned h = (unsigned)(mant >> 32) + ((unsigned)(1022 + 31 - lz) << 20);
  return __hiloint2double(a ? (int)(h | ((unsigned)n & 0x80000000u)) : 0, (int)(unsigned)mant);
}
__device__ __forceinline__ float floor_int(float v, unsigned& k) {
  const float f = floorf(v);
  k = (unsigned)(int)f;
  return f;
}

// Spectral layout of the state: columns per tile, and the element of (ky_idx, kx).
template <typename T> __host__ __device__ constexpr int spec_tile() { return sizeof(T) == 4 ? 4 : 2; }
template <typename T> __host__ __device__ __forceinline__ int spec_index(int kyi, int kx, int NY) {
  constexpr int S = sizeof(T) == 4 ? 4 : 2;
  return (kx / S) * (NY * S) + kyi * S + kx % S;
}

// Global loads and stores of memory that the kernels of a step hand to one
// another.  A stage kernel is resident while the previous one still writes (see
// pdl_wait), so nothing that a kernel of the step writes may be read through the
// read-only path (__ldg, or loads that the compiler may take for such): that
// path is for data no kernel writes while this one lives (run descriptors,
// tables).  The compiler keeps these accesses in order with one another and
// with pdl_wait, and does not treat them as touching other memory: after a
// plain store through a pointer it would reload every run-descriptor field it
// uses (kept in shared memory), a chain of waits per store.  Values handed from
// one thread of a block to another through them need a __syncthreads between
// the store and the load (the split column blocks' u, v and h).
__device__ __forceinline__ void gst(float2* p, float2 v) {
  asm volatile("st.global.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(v.x), "f"(v.y));
}
__device__ __forceinline__ void gst(double2* p, double2 v) {
  asm volatile("st.global.v2.f64 [%0], {%1, %2};" ::"l"(p), "d"(v.x), "d"(v.y));
}
__device__ __forceinline__ float gld(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ double gld(const double* p) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float2 gld(const float2* p) {
  float2 v;
  asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ double2 gld(const double2* p) {
  double2 v;
  asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 gld(const float4* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
// The two rows of a pair at one kx of a mixed field.
__device__ __forceinline__ void ld_pair(const float2* p, float2& a, float2& b) {
  const float4 v = gld(reinterpret_cast<const float4*>(p));
  a = make_float2(v.x, v.y);
  b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void ld_pair(const double2* p, double2& a, double2& b) {
  a = gld(p);
  b = gld(p + 1);
}
__device__ __forceinline__ void st_pair(float2* p, float2 a, float2 b) {
  *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st_pair(double2* p, double2 a, double2 b) {
  p[0] = a;
  p[1] = b;
}

// Distance between the transforms of a block (rows, or the columns of a
// column tile).
template <typename T>
__host__ __device__ __forceinline__ int row_stride(int N) { return N + (N >> 3); }
template <typename T>
__host__ __device__ __forceinline__ int col_stride(int N, int C) { return N + (N >> 3); }
// Column tiles on group transforms (lanes interleave the C columns): each
// column owns two exchange buffers, and successive columns are offset by a
// number of slots (16 for FP32, 8 for FP64, per bank row) congruent to
// slots/C, so the C lanes that share a row index use distinct slots.
template <typename T>
__host__ __device__ __forceinline__ int col_buf_stride(int N, int C) {
  const int S = sizeof(T) == 4 ? 16 : 8;
  const int st = 2 * (N + (N >> 3));
  const int tgt = C <= S ? S / C : 1;
  return st + (((tgt - st) % S) + S) % S;
}

// ---------------------------------------------------------------------------
// Geometry of one grid
struct Geom {
  int N, log2N, K, KX, KXP, NY;
  long long ms;  // complex elements per spectral field  (NY * KXP)
  long long mi;  // complex elements per mixed field     (N * KXP)
  long long np;  // reals per physical field             (N * N)
};

// ---------------------------------------------------------------------------
// Field bookkeeping for one configuration (strategy, mask) of a handle.
enum { MAXF = 16, MAXI = 24, MAXP = 16 };
enum { OP_ID = 0, OP_DX = 1, OP_DY = 2, OP_CURL = 3 };
enum { LMF_ZETA = 0, LMF_H = 1, LMF_U = 2, LMF_V = 3, LMF_Q = 4, NLMF = 5 };
// physical fields of the row pass (and of the Strategy-2 gather buffer)
enum { PH_U = 0, PH_V = 1, PH_H = 2, PH_Z = 3, PH_Q = 4, PH_XX = 5, PH_XY = 6, NPH = 7 };
// products formed in physical space by the row pass
enum {
  PK_ZV = 0,   // zeta v
  PK_ZU = 1,   // zeta u
  PK_KE = 2,   // (u^2 + v^2)/2
  PK_HU = 3,   // h u
  PK_HV = 4,   // h v
  PK_Q = 5,    // (f0 + zeta)/h
  PK_ADV = 6,  // u d_x G + v d_y G            (Strategy 1; a, b: mixed d_x G, d_y G)
  PK_XI = 7,   // u_c(x+xi) - w_c - w.grad xi_c (Strategy 2; c: component)
  PK_GBAR = 8  // f(x+xi) - w.grad g           (Strategy 2; c: PH_* of f)
};
// integrating-factor classes
enum { IF_DYN = 0, IF_LM = 1, IF_NONE = 2 };
// tasks of the column-stage kernel (see k_stage_col)
enum { CT_UV = 0, CT_E2 = 1, CT_KIN = 2, CT_H = 3, CT_G = 4, CT_P = 5, MAXCT = 10 };
// A task's steps, in order: with op < 0 the forward transform of product
// `prod` (-1: none, the values are there), whose result is kept (CA_KEEP),
// parked (CA_PARK) or updates field `fld` (CA_U and CA_V: u and v of CT_UV;
// CA_UPD; CA_UPD_PARK: the new value is parked too); with op = OP_* the inverse
// transform of op(value) into mixed field `prod`, the value being what the
// update before left (CA_X), the parked one (CA_PARKED) or that of field `fld`
// in memory (CA_MEM).  part: which part of the block takes the step when the
// block is split in halves or quarters; bar: a block barrier comes before it then.
enum {
  CA_PARK = 0, CA_U = 1, CA_V = 2, CA_UPD = 3, CA_UPD_PARK = 4, CA_X = 5, CA_PARKED = 6, CA_MEM = 7, CA_KEEP = 8,
  MAXCS = 8
};
// (Bytes: the descriptor is part of the column stage's static shared memory,
// which at 2048^2 in FP32 has to stay below 196 KB with the buffers: above it
// the SM's L1 shrinks from 60 to 28 KB, 245 -> 283 us.)
struct ColTask {
  signed char kind, slot;  // CT_*; mean-field slot or component
  signed char n;
  signed char prod[MAXCS], act[MAXCS], op[MAXCS], fld[MAXCS], part[MAXCS], bar[MAXCS];
};
// role of an evolved field in the right-hand side
enum { R_U = 0, R_V = 1, R_H = 2, R_G = 3, R_P = 4, R_E = 5 };

struct Layout {
  int strategy;   // 0: dynamics only, 1 or 2
  int scheme;     // SCHEME_* (the C ABI's LM_SCHEME_*) of the open interval
  int model;      // 0 shallow water, 1 kinematic
  int nf;         // evolved spectral fields
  int ni;         // mixed intermediates produced by the column pass
  int np;         // product fields produced by the row pass
  int nlm;        // number of Lagrangian-mean scalar fields
  int lmf[NLMF];  // which scalar (LMF_*) each LM slot averages
  int has_pos, eulerian, has_q;
  // evolved-field indices
  int f_u, f_v, f_h;
  int f_g[NLMF];     // g~ (S1) or gbar (S2) per LM slot
  int f_p[2];        // D (S1) or xi (S2) components
  int f_e[NLMF];     // Eulerian accumulators per LM slot
  int fclass[MAXF];  // IF_* class of each evolved field
  int fkahan[MAXF];  // compensated final update (FP32 mode) for this field
  int frole[MAXF];   // R_* role
  // column pass: output i = op(src[i] (, src2[i]))
  int i_src[MAXI], i_src2[MAXI], i_op[MAXI];
  int i_u, i_v, i_h, i_z;      // dynamics intermediates
  int i_xi[2];                 // xi components (Strategy 2)
  // row pass: product list
  int pk[MAXP], pa[MAXP], pb[MAXP], pc[MAXP];
  // product index feeding each right-hand side (-1: none)
  int p_zv, p_zu, p_ke, p_hu, p_hv, p_q;
  int p_g[NLMF];
  int p_p[2];
  // tasks of the column-stage kernel
  int nct;
  ColTask ct[MAXCT];
};

// discretisation of the mean equations (the C ABI's LM_SCHEME_* values)
enum { SCHEME_COUPLED = 0, SCHEME_XI_FIRST = 1 };

struct StepConsts {
  double dt, f0, c2, adv_x, adv_y;
  int stepper;  // SW_STEP_* (0 RK4, 1 Heun, 2 forward Euler)
  int pad;
};

// Programmatic dependent launch (PTX griddepcontrol).  The stage kernels of
// a step are launched with programmatic stream serialisation, so a kernel's
// blocks may start while the previous kernel of the stream finishes.
// pdl_wait: before its first access to memory that earlier kernels write,
// a stage kernel waits until they have completed and their writes are
// visible (without the launch attribute it returns at once).  pdl_release,
// right after it: once every block of this kernel has started, the next
// kernel's blocks may take what is free on the SMs, read their run
// descriptors (which no kernel writes) and wait in turn.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// passes of the stage pipeline per step of a stepper: RK4 4 stages, Heun 2,
// forward Euler 1 stage and an update-only pass that commits y_{n+1}
__host__ __device__ __forceinline__ int stage_count(int stepper) { return stepper == 0 ? 4 : 2; }

}  // namespace lm
