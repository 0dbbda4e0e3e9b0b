// launch.cuh -- host-side launchers for the kernels of kernels.cuh and
// stage.cuh.  Instantiated once per precision (kernels_f32.cu, kernels_f64.cu).
#pragma once
#include <string>

#include "stage.cuh"

struct sw_handle;

namespace lm {

// Rows (row pairs in the stage kernels) per block: B of N points run with
// B*N/8 threads (one 8-element Stockham butterfly set per thread and pass);
// `points` = B*N.
inline int row_block_rows(int N, int points = 512) {
  int B = points / N;
  if (B > N) B = N;
  if (B < 1) B = 1;
  return B;
}
// Row pairs per block of the stage kernels: at most N/2, but a warp's worth of
// threads (at N = 16 the pairs then wrap around, each done twice).
inline int row_block_pairs(int N, int points) {
  int B = row_block_rows(N, points);
  if (B > N / 2) B = N / 2;
  return B * N < 256 ? 256 / N : B;
}
inline int row_blocks(int N, int B) { return N / 2 > B ? N / 2 / B : 1; }

// Row pass: B row pairs per block, W groups of N/8 threads per pair (see
// k_stage_row_prod); the block may hold up to row_prod_max_threads threads.
template <typename T> bool row_prod_fused(int N, const Layout& L) {
  // FP64 from 1024^2 the base fields take 64 KB and more per row pair and leave
  // one block per SM: row pass alone 419 us with them, 299 us + 54 us for the
  // planes.  FP32: 250 us against 349 us + 39 us at 2048^2.
  return L.strategy != 2 && (sizeof(T) == 4 || N <= 512);
}
// Strategy 2: the gathered arrays within 96 KB per row pair.
template <typename T> bool row_prod_gath(int N, const Layout& L) {
  return L.strategy == 2 && (size_t)row_prod_planes(0, 1, L.has_q) * N * sizeof(cplx<T>) <= (size_t)96 * 1024;
}
template <typename T> size_t row_prod_smem(int N, int B, int W, const Layout& L, bool all_products = true) {
  const size_t nu = row_prod_planes(row_prod_fused<T>(N, L), all_products && row_prod_gath<T>(N, L), L.has_q);
  return (size_t)B * sizeof(cplx<T>) * (nu * N + (size_t)W * 2 * row_stride<T>(N));
}

// Largest W for B row pairs and np products per block (other than a team): W > 1 needs whole
// warps per group (N >= 256), a thread count within the block limit, at most
// 15 named barriers (groups of N >= 512) and at most 200 KB of shared memory.
template <typename T> int row_prod_groups(int N, int B, int np, const Layout& L, bool alone) {
  const int G = N / 8;
  if (G < 32) return 1;
  auto fit = [&](int threads, size_t smem) {
    int W = np < 1 ? 1 : np;
    while (W > 1 && (B * W * G > threads || (G >= 64 && B * W > 15) || row_prod_smem<T>(N, B, W, L) > smem)) --W;
    return W;
  };
  // two blocks per SM, or one of several groups where that leaves one group or,
  // FP32, the launch has no second block for an SM anyway (`alone`; 256^2, Strategy 2
  // with PV, 13 products: 12 -> 13 groups, a step 115 -> 107 us)
  const int W = fit(sizeof(T) == 4 ? 384 : 256, (size_t)110 * 1024);
  return W > 1 && !(alone && sizeof(T) == 4) ? W : fit(row_prod_max_threads<T>(), (size_t)200 * 1024);
}

// Row pairs per block of the row inverse pass.
inline int row_inv_pairs(int N, int points) { return row_block_pairs(N, points > 512 ? points : 512); }

// Row passes by teams of four sets of groups per row pair (see
// k_stage_row_prod): one product per block, groups within a warp, few enough row
// pairs for the block, and all blocks resident at once, row_team_blocks() per SM (by
// registers), since a team's blocks hold four times the warps.  A step, without -> with
// teams: FP64 16^2 Strategy 2 239 -> 173 us, 64^2 Strategy 1 168 -> 141, four 64^2 runs 191 ->
// 157; FP32 64^2 Strategy 1 54 -> 45.  Beyond: 16 64^2 runs' dynamics in FP64 (640 blocks)
// 166 against 180, 32 in FP32 (1280) 68 against 76.
template <typename T> constexpr int row_team_blocks() { return sizeof(T) == 4 ? 6 : 4; }
template <typename T> bool row_team(int N, int points, int ppb) {
  const int G = N / 8;
  return G < 32 && ppb == 1 && 4 * row_block_pairs(N, points) * G <= row_prod_max_threads<T>() &&
         4 * row_inv_pairs(N, points) * G <= 256;
}

template <typename T> constexpr int SPLIT_THREADS() { return sizeof(T) == 4 ? 256 : 128; }

// one field at a time, without device memory of their own (csrc/project_static.cu)
template <typename T> cudaError_t launch_col_inv(const ColArgs<T>& a, cudaStream_t s);
template <typename T> cudaError_t launch_col_fwd(const ColArgs<T>& a, cudaStream_t s);
template <typename T> cudaError_t launch_row_inv(const RowInvArgs<T>& a, cudaStream_t s);
template <typename T> cudaError_t launch_row_fwd(const RowFwdArgs<T>& a, cudaStream_t s);
// parts: into how many the column stage's blocks are split (2 and 4: at most
// SPLIT_THREADS threads).
// warp: every run's rows have N <= 256 (groups of at most one warp), so the
// row kernels' variant without named barriers may run.  pdl: launch with
// programmatic stream serialisation (see pdl_wait).
template <typename T>
cudaError_t launch_stage(int kt, const RunDesc<T>* runs, const int* start, int nruns, int blocks, int threads,
                         size_t smem, int stage, bool warp, int parts, bool pdl, cudaStream_t s);
// FP64 transforms between the state and physical planes (see k_out_col).
template <typename T> cudaError_t launch_out(const OutArgs<T>& a, cudaStream_t s);
template <typename T> cudaError_t launch_in(const InArgs<T>& a, cudaStream_t s);
template <typename T>
cudaError_t launch_spec_rows(cplx<T>* t0, cplx<T>* t1, cplx<T>* rows, const Geom& g, int nf, bool to_rows,
                             long long* ctr, long long done, cudaStream_t s);
template <typename T>
cudaError_t launch_velocity_from_vorticity(cplx<T>* y, const Geom& g, int fu, int fv, int fh, cudaStream_t s);
cudaError_t launch_diag(const double* phys, long long np, double f0, double c2, double* part, int nblk,
                        double* out, cudaStream_t s);
cudaError_t launch_spectrum_shells(const double2* F, const Geom& g, double* acc, cudaStream_t s);

// Handle hooks for other translation units (defined in lagmean.cu).
struct HandleInfo {
  int N, model;
  double dt, f0, adv_x, adv_y;
  bool lm_open;
  cudaStream_t stream;
};
int handle_info(sw_handle* h, HandleInfo* hi);
// FP64 physical u, v, h, zeta of the state (4 * N * N doubles in the handle's
// staging buffer, valid until the handle's next call), on its stream
int handle_phys_uvhz(sw_handle* h, const double** out);
void handle_set_error(sw_handle* h, const std::string& msg);

#ifdef LM_INSTANTIATE
// Raise the dynamic shared-memory limit of every kernel once (outside any
// stream capture), to the device's opt-in maximum.
template <typename K> static cudaError_t allow_dynamic_smem(K kern, int optin) {
  // static and dynamic shared memory together may not exceed the opt-in limit
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, kern);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
}

template <typename T> static cudaError_t prepare_kernels_t() {
  int dev = 0, mx = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&mx, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
  if constexpr (sizeof(T) == 8) {
    if ((e = allow_dynamic_smem(k_col_inv<T>, mx)) != cudaSuccess) return e;
    if ((e = allow_dynamic_smem(k_col_fwd<T>, mx)) != cudaSuccess) return e;
    if ((e = allow_dynamic_smem(k_row_inv<T>, mx)) != cudaSuccess) return e;
    if ((e = allow_dynamic_smem(k_row_fwd<T>, mx)) != cudaSuccess) return e;
  }
  if ((e = allow_dynamic_smem(k_out_col<T>, mx)) != cudaSuccess) return e;
  if ((e = allow_dynamic_smem(k_out_row<T>, mx)) != cudaSuccess) return e;
  if ((e = allow_dynamic_smem(k_in_row<T>, mx)) != cudaSuccess) return e;
  if ((e = allow_dynamic_smem(k_in_col<T>, mx)) != cudaSuccess) return e;
  if constexpr (sizeof(T) == 8)
    if ((e = allow_dynamic_smem(k_stage_col<T, 128, 1>, mx)) != cudaSuccess) return e;
  if ((e = allow_dynamic_smem(k_stage_col<T, 256, 1>, mx)) != cudaSuccess) return e;
  if ((e = allow_dynamic_smem(k_stage_col<T, SPLIT_THREADS<T>(), 2>, mx)) != cudaSuccess) return e;
  if ((e = allow_dynamic_smem(k_stage_col<T, SPLIT_THREADS<T>(), 4>, mx)) != cudaSuccess) return e;
  if constexpr (sizeof(T) == 4) {
    if ((e = allow_dynamic_smem(k_stage_col<T, 512, 1>, mx)) != cudaSuccess) return e;
    if ((e = allow_dynamic_smem(k_stage_col<T, 1024, 1>, mx)) != cudaSuccess) return e;
  }
  if ((e = allow_dynamic_smem(k_stage_row_inv<T, false>, mx)) != cudaSuccess) return e;
  if ((e = allow_dynamic_smem(k_stage_row_inv<T, true>, mx)) != cudaSuccess) return e;
  if ((e = allow_dynamic_smem(k_stage_row_prod<T, false>, mx)) != cudaSuccess) return e;
  if ((e = allow_dynamic_smem(k_stage_row_prod<T, true>, mx)) != cudaSuccess) return e;
  return cudaSuccess;
}

template <typename T> cudaError_t launch_col_inv(const ColArgs<T>& a, cudaStream_t s) {
  const size_t sm = (size_t)4 * col_stride<T>(a.g.N, 4) * sizeof(cplx<T>);
  k_col_inv<T><<<a.g.KXP / 4, a.g.N / 2, sm, s>>>(a);
  return cudaGetLastError();
}

template <typename T> cudaError_t launch_col_fwd(const ColArgs<T>& a, cudaStream_t s) {
  const size_t sm = (size_t)4 * col_stride<T>(a.g.N, 4) * sizeof(cplx<T>);
  k_col_fwd<T><<<a.g.KXP / 4, a.g.N / 2, sm, s>>>(a);
  return cudaGetLastError();
}

template <typename T> cudaError_t launch_row_inv(const RowInvArgs<T>& a, cudaStream_t s) {
  const size_t sm = (size_t)a.B * row_stride<T>(a.g.N) * sizeof(cplx<T>);
  k_row_inv<T><<<a.g.N / a.B, a.B * a.g.N / 8, sm, s>>>(a);
  return cudaGetLastError();
}

template <typename T> cudaError_t launch_row_fwd(const RowFwdArgs<T>& a, cudaStream_t s) {
  const size_t sm = (size_t)a.B * row_stride<T>(a.g.N) * sizeof(cplx<T>);
  k_row_fwd<T><<<a.g.N / a.B, a.B * a.g.N / 8, sm, s>>>(a);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_stage(int kt, const RunDesc<T>* runs, const int* start, int nruns, int blocks, int threads,
                         size_t smem, int stage, bool warp, int parts, bool pdl, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  switch (kt) {
    case KT_ROW_INV:
      return warp ? cudaLaunchKernelEx(&cfg, k_stage_row_inv<T, true>, runs, start, nruns)
                  : cudaLaunchKernelEx(&cfg, k_stage_row_inv<T, false>, runs, start, nruns);
    case KT_ROW_PROD:
      return warp ? cudaLaunchKernelEx(&cfg, k_stage_row_prod<T, true>, runs, start, nruns, stage)
                  : cudaLaunchKernelEx(&cfg, k_stage_row_prod<T, false>, runs, start, nruns, stage);
    case KT_KIN:
      return cudaLaunchKernelEx(&cfg, k_stage_kin<T>, runs, start, nruns, stage);
    default:
      if (parts == 4) return cudaLaunchKernelEx(&cfg, k_stage_col<T, SPLIT_THREADS<T>(), 4>, runs, start, nruns, stage);
      if (parts == 2) return cudaLaunchKernelEx(&cfg, k_stage_col<T, SPLIT_THREADS<T>(), 2>, runs, start, nruns, stage);
      if constexpr (sizeof(T) == 4) {
        if (threads > 512) return cudaLaunchKernelEx(&cfg, k_stage_col<T, 1024, 1>, runs, start, nruns, stage);
        if (threads > 256) return cudaLaunchKernelEx(&cfg, k_stage_col<T, 512, 1>, runs, start, nruns, stage);
      }
      if constexpr (sizeof(T) == 8)
        if (threads <= 128) return cudaLaunchKernelEx(&cfg, k_stage_col<T, 128, 1>, runs, start, nruns, stage);
      return cudaLaunchKernelEx(&cfg, k_stage_col<T, 256, 1>, runs, start, nruns, stage);
  }
}

struct IoShape {
  dim3 cols, rows;
  int cthr, rthr;
  size_t csm, rsm;
  IoShape(const Geom& g, int n) {
    const int lC = io_log2C(g.N), B = row_block_pairs(g.N, 512);
    cols = dim3((unsigned)(g.KXP >> lC), (unsigned)n);
    rows = dim3((unsigned)row_blocks(g.N, B), (unsigned)n);
    cthr = (g.N << lC) / 8;
    rthr = B * g.N / 8;
    csm = ((size_t)col_buf_stride<double>(g.N, 1 << lC) << lC) * sizeof(double2);
    rsm = (size_t)B * 2 * row_stride<double>(g.N) * sizeof(double2);
  }
};
template <typename T> cudaError_t launch_out(const OutArgs<T>& a, cudaStream_t s) {
  const IoShape q(a.g, a.n);
  k_out_col<T><<<q.cols, q.cthr, q.csm, s>>>(a);
  k_out_row<T><<<q.rows, q.rthr, q.rsm, s>>>(a);
  return cudaGetLastError();
}
template <typename T> cudaError_t launch_in(const InArgs<T>& a, cudaStream_t s) {
  const IoShape q(a.g, a.n);
  k_in_row<T><<<q.rows, q.rthr, q.rsm, s>>>(a);
  k_in_col<T><<<q.cols, q.cthr, q.csm, s>>>(a);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_spec_rows(cplx<T>* t0, cplx<T>* t1, cplx<T>* rows, const Geom& g, int nf, bool to_rows,
                             long long* ctr, long long done, cudaStream_t s) {
  k_spec_rows<T><<<(unsigned)((g.ms * 2 * nf + 255) / 256), 256, 0, s>>>(t0, t1, rows, g, nf, to_rows ? 1 : 0, ctr, done);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_velocity_from_vorticity(cplx<T>* y, const Geom& g, int fu, int fv, int fh, cudaStream_t s) {
  k_velocity_from_vorticity<T><<<(unsigned)((g.ms + 255) / 256), 256, 0, s>>>(y, g, fu, fv, fh);
  return cudaGetLastError();
}

#define LM_INSTANTIATE_ALL(T)                                                                               \
  template cudaError_t launch_stage<T>(int, const RunDesc<T>*, const int*, int, int, int, size_t, int, bool,  \
                                       int, bool, cudaStream_t);                                            \
  template cudaError_t launch_out<T>(const OutArgs<T>&, cudaStream_t);                                       \
  template cudaError_t launch_in<T>(const InArgs<T>&, cudaStream_t);                                         \
  template cudaError_t launch_spec_rows<T>(cplx<T>*, cplx<T>*, cplx<T>*, const Geom&, int, bool, long long*, long long,   \
                                           cudaStream_t);                                                    \
  template cudaError_t launch_velocity_from_vorticity<T>(cplx<T>*, const Geom&, int, int, int, cudaStream_t);
// the generic FP64 transforms (csrc/project_static.cu)
#define LM_INSTANTIATE_GENERIC                                                                              \
  template cudaError_t launch_col_inv<double>(const ColArgs<double>&, cudaStream_t);                         \
  template cudaError_t launch_col_fwd<double>(const ColArgs<double>&, cudaStream_t);                         \
  template cudaError_t launch_row_inv<double>(const RowInvArgs<double>&, cudaStream_t);                      \
  template cudaError_t launch_row_fwd<double>(const RowFwdArgs<double>&, cudaStream_t);
#endif

}  // namespace lm
