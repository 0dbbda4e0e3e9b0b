// lagmean.cu -- C ABI (include/lagmean.h): handles, field layout, the RK4
// stage pipeline replayed from a captured CUDA graph, and the FP64 transforms
// around it (initial condition, end-of-interval means, diagnostics).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>

#include <vector>

#include "../../include/lagmean.h"
#include "launch.cuh"

using namespace lm;

namespace lm {
cudaError_t prepare_kernels_f32();
cudaError_t prepare_kernels_f64();
}  // namespace lm

static thread_local std::string g_create_error;

namespace lm {
// message for calls without a handle (sw_create, sw_project_static)
void set_handleless_error(const std::string& msg) { g_create_error = msg; }
}  // namespace lm

struct BatchExec;

struct sw_handle {
  sw_params p;
  Geom g;
  cudaStream_t stream = nullptr;
  bool fp32 = false;
  size_t tsz = 8;  // sizeof(T)
  std::string err;
  // device memory
  void* arena = nullptr;
  size_t arena_bytes = 0;
  void *y = nullptr, *ys = nullptr, *ys2 = nullptr, *acc = nullptr, *comp = nullptr;
  void *mix = nullptr, *pmix = nullptr, *phys = nullptr, *ef = nullptr, *tw = nullptr;
  TwFx* tw64 = nullptr;
  double2 *spec64 = nullptr, *mix64 = nullptr;
  double *out64 = nullptr, *part = nullptr, *dres = nullptr;
  long long* ctr = nullptr;
  unsigned* ticket = nullptr;
  int diag_blocks = 0;
  // interval state
  bool lm_open = false;
  lm_params lp{};
  int64_t done = 0;
  int64_t steps_total = 0;
  Layout L{};
  // launch shapes: column tiles of at most 2^lC columns; row_prod `points`
  // per block (row pairs x N) and ppb products per block (0: automatic, see
  // batch_build_t)
  int lC = 2, points = 256, ppb = 0;
  uint64_t version = 1;  // bumped whenever L or the launch shapes change
  BatchExec* self = nullptr;  // batch of one used by sw_step / lmean_step
  int64_t launches = 0;  // kernels launched since creation
};

static int fail(sw_handle* h, int code, const std::string& msg) {
  if (h) h->err = msg;
  else g_create_error = msg;
  return code;
}
static int fail_cuda(sw_handle* h, const char* what, cudaError_t e) {
  return fail(h, SW_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}
#define CK(h, ...)                                                  \
  do {                                                              \
    cudaError_t e_ = (__VA_ARGS__);                                 \
    if (e_ != cudaSuccess) return fail_cuda(h, #__VA_ARGS__, e_);   \
  } while (0)

// ---------------------------------------------------------------------------
// Field layout of a configuration.
static_assert(SCHEME_COUPLED == LM_SCHEME_COUPLED && SCHEME_XI_FIRST == LM_SCHEME_XI_FIRST, "scheme values");

static Layout build_layout(const sw_params& p, int strategy, int fields, int eulerian, int scheme = 0) {
  Layout L;
  std::memset(&L, 0, sizeof(L));
  L.strategy = strategy;
  L.scheme = scheme;
  L.model = p.model;
  L.p_zv = L.p_zu = L.p_ke = L.p_hu = L.p_hv = L.p_q = -1;
  for (int j = 0; j < NLMF; ++j) L.f_g[j] = L.f_e[j] = L.p_g[j] = -1;
  L.f_p[0] = L.f_p[1] = L.p_p[0] = L.p_p[1] = L.i_xi[0] = L.i_xi[1] = -1;
  int nf = 0;
  L.f_u = nf++;
  L.f_v = nf++;
  L.f_h = nf++;
  for (int f = 0; f < 3; ++f) {
    // the Laplacian acts on momentum only (Eq. sw_momentum_dimless; the mass
    // equation has no viscous term), the hyperviscosity on u, v and h
    L.fclass[f] = (f == 2 && p.visc == SW_VISC_LAPLACE) ? IF_NONE : IF_DYN;
    L.fkahan[f] = 0;
    L.frole[f] = R_U + f;
  }
  if (strategy > 0) {
    const int bits[NLMF] = {LM_ZETA, LM_H, LM_U, LM_V, LM_Q};
    for (int j = 0; j < NLMF; ++j)
      if (fields & bits[j]) L.lmf[L.nlm++] = j;
    L.has_q = (fields & LM_Q) ? 1 : 0;
    L.has_pos = (strategy == 2 || (fields & LM_POS)) ? 1 : 0;
    L.eulerian = eulerian ? 1 : 0;
    auto addf = [&](int cls, int role) {
      L.fclass[nf] = cls;
      L.fkahan[nf] = 1;
      L.frole[nf] = role;
      return nf++;
    };
    for (int j = 0; j < L.nlm; ++j) L.f_g[j] = addf(IF_LM, R_G);
    if (L.has_pos)
      for (int c = 0; c < 2; ++c) L.f_p[c] = addf(IF_LM, R_P);
    if (L.eulerian)
      for (int j = 0; j < L.nlm; ++j) L.f_e[j] = addf(IF_NONE, R_E);
  }
  L.nf = nf;
  // column-pass outputs
  int ni = 0;
  auto addi = [&](int src, int op, int src2) {
    L.i_src[ni] = src;
    L.i_op[ni] = op;
    L.i_src2[ni] = src2;
    return ni++;
  };
  L.i_u = addi(L.f_u, OP_ID, -1);
  L.i_v = addi(L.f_v, OP_ID, -1);
  L.i_h = addi(L.f_h, OP_ID, -1);
  // the two-dimensional Euler model evolves zeta itself (the h slot; its
  // mean, which a curl of u would drop, included)
  L.i_z = p.model == SW_MODEL_EULER2D ? L.i_h : addi(L.f_u, OP_CURL, L.f_v);
  // products
  int np = 0;
  auto addp = [&](int kind, int a, int b, int c) {
    L.pk[np] = kind;
    L.pa[np] = a;
    L.pb[np] = b;
    L.pc[np] = c;
    return np++;
  };
  if (p.model == SW_MODEL_SW) {
    L.p_zv = addp(PK_ZV, -1, -1, 0);
    L.p_zu = addp(PK_ZU, -1, -1, 0);
    L.p_ke = addp(PK_KE, -1, -1, 0);
    L.p_hu = addp(PK_HU, -1, -1, 0);
    L.p_hv = addp(PK_HV, -1, -1, 0);
  } else if (p.model == SW_MODEL_EULER2D) {
    // zeta v and zeta u: d_t zeta = -d_x (u zeta) - d_y (v zeta)
    L.p_zv = addp(PK_ZV, -1, -1, 0);
    L.p_zu = addp(PK_ZU, -1, -1, 0);
  }
  if (L.has_q) L.p_q = addp(PK_Q, -1, -1, 0);
  const int ph_of[NLMF] = {PH_Z, PH_H, PH_U, PH_V, PH_Q};
  if (strategy == 1) {
    for (int j = 0; j < L.nlm; ++j) {
      const int gx = addi(L.f_g[j], OP_DX, -1), gy = addi(L.f_g[j], OP_DY, -1);
      L.p_g[j] = addp(PK_ADV, gx, gy, 0);
    }
    if (L.has_pos)
      for (int c = 0; c < 2; ++c) {
        const int dx = addi(L.f_p[c], OP_DX, -1), dy = addi(L.f_p[c], OP_DY, -1);
        L.p_p[c] = addp(PK_ADV, dx, dy, 0);
      }
  } else if (strategy == 2) {
    L.i_xi[0] = addi(L.f_p[0], OP_ID, -1);
    L.i_xi[1] = addi(L.f_p[1], OP_ID, -1);
    for (int c = 0; c < 2; ++c) {
      const int dx = addi(L.f_p[c], OP_DX, -1), dy = addi(L.f_p[c], OP_DY, -1);
      L.p_p[c] = addp(PK_XI, dx, dy, c);
    }
    for (int j = 0; j < L.nlm; ++j) {
      const int gx = addi(L.f_g[j], OP_DX, -1), gy = addi(L.f_g[j], OP_DY, -1);
      L.p_g[j] = addp(PK_GBAR, gx, gy, ph_of[L.lmf[j]]);
    }
  }
  // Products that need transforms of their own (advection, Strategy 2) first:
  // the row pass's groups take products in this order.
  {
    auto heavy = [](int k) { return k == PK_ADV || k == PK_XI || k == PK_GBAR; };
    int pos[MAXP], no = 0;
    const Layout Q = L;
    for (int pass = 0; pass < 2; ++pass)
      for (int q = 0; q < np; ++q)
        if (heavy(Q.pk[q]) == (pass == 0)) {
          pos[q] = no;
          L.pk[no] = Q.pk[q];
          L.pa[no] = Q.pa[q];
          L.pb[no] = Q.pb[q];
          L.pc[no++] = Q.pc[q];
        }
    auto remap = [&](int& idx) {
      if (idx >= 0) idx = pos[idx];
    };
    remap(L.p_zv);
    remap(L.p_zu);
    remap(L.p_ke);
    remap(L.p_hu);
    remap(L.p_hv);
    remap(L.p_q);
    for (int j = 0; j < NLMF; ++j) remap(L.p_g[j]);
    remap(L.p_p[0]);
    remap(L.p_p[1]);
  }
  L.ni = ni;
  L.np = np;
  return L;
}

// Tasks of the column-stage kernel (the longest first) for whole blocks or
// for blocks split in `parts` = 2 or 4 parts.
static void build_tasks(Layout& L, int parts) {
  std::memset(L.ct, 0, sizeof(L.ct));
  L.nct = 0;
  const bool split = parts > 1, quad = parts == 4;
  ColTask* t = nullptr;
  auto task = [&](int kind, int slot) {
    t = &L.ct[L.nct++];
    t->kind = (signed char)kind;
    t->slot = (signed char)slot;
  };
  auto step = [&](int prod, int act, int op, int fld, int part = 0, int bar = 0) {
    const int i = t->n++;
    t->prod[i] = (signed char)prod;
    t->act[i] = (signed char)act;
    t->op[i] = (signed char)op;
    t->fld[i] = (signed char)fld;
    t->part[i] = (signed char)part;
    t->bar[i] = (signed char)bar;
  };
  if (L.model == SW_MODEL_SW) {
    task(CT_UV, 0);
    step(L.p_ke, CA_PARK, -1, -1);
    if (quad) {
      step(L.p_zv, CA_KEEP, -1, -1, 1);
      step(L.p_zu, CA_KEEP, -1, -1, 2);
      step(-1, CA_U, -1, L.f_u, 1, 1);
      step(-1, CA_V, -1, L.f_v, 2);
      step(L.i_z, CA_MEM, OP_CURL, L.f_u, 0, 1);
      step(L.i_u, CA_X, OP_ID, L.f_u, 1);
      step(L.i_v, CA_X, OP_ID, L.f_v, 2);
    } else if (split) {
      step(L.p_zu, CA_KEEP, -1, -1, 1);
      step(L.p_zv, CA_U, -1, L.f_u, 0, 1);
      step(-1, CA_V, -1, L.f_v, 1);
      step(L.i_v, CA_X, OP_ID, L.f_v, 1);
      step(L.i_u, CA_X, OP_ID, L.f_u, 0, 1);
      step(L.i_z, CA_MEM, OP_CURL, L.f_u, 1);
    } else {
      step(L.p_zv, CA_U, -1, L.f_u);
      step(L.i_u, CA_X, OP_ID, L.f_u);
      step(L.p_zu, CA_V, -1, L.f_v);
      step(L.i_v, CA_X, OP_ID, L.f_v);
      step(L.i_z, CA_MEM, OP_CURL, L.f_u);
    }
  } else if (L.model == SW_MODEL_EULER2D) {
    task(CT_E2, 0);
    step(L.p_zu, CA_PARK, -1, -1);
    if (split) step(L.p_zv, CA_KEEP, -1, -1, 1);
    step(split ? -1 : L.p_zv, CA_UPD, -1, L.f_h, 1, 1);
    step(L.i_h, CA_X, OP_ID, L.f_h, 1, 1);
    step(L.i_u, CA_MEM, OP_ID, L.f_u);
    step(L.i_v, CA_MEM, OP_ID, L.f_v, quad ? 2 : 0);
  } else {
    task(CT_KIN, 0);
    for (int f = 0; f < 3; ++f) step(-1, CA_UPD, -1, f, quad ? f : 0);
    step(L.i_h, CA_MEM, OP_ID, L.f_h, quad ? 2 : 0, 1);
    step(L.i_z, CA_MEM, OP_CURL, L.f_u, quad ? 3 : 0);
    step(L.i_u, CA_MEM, OP_ID, L.f_u, quad ? 0 : 1);
    step(L.i_v, CA_MEM, OP_ID, L.f_v, 1);
  }
  if (L.has_pos)
    for (int c = 0; c < 2; ++c) {
      const int q = L.p_p[c];
      task(CT_P, c);
      step(q, CA_UPD_PARK, -1, L.f_p[c]);
      if (L.strategy == 2) {
        step(L.i_xi[c], CA_X, OP_ID, L.f_p[c], 0, 1);
        step(L.pa[q], CA_PARKED, OP_DX, L.f_p[c], quad ? 2 : 0);
      } else {
        step(L.pa[q], CA_X, OP_DX, L.f_p[c], 0, 1);
      }
      step(L.pb[q], CA_PARKED, OP_DY, L.f_p[c], 1);
    }
  for (int j = 0; j < L.nlm; ++j) {
    const int q = L.p_g[j];
    task(CT_G, j);
    const bool apart = quad && L.lmf[j] == LMF_Q;  // q's transform beside the product's
    if (L.lmf[j] == LMF_Q) step(L.p_q, CA_PARK, -1, -1, apart ? 1 : 0);
    if (apart) step(q, CA_KEEP, -1, -1);
    step(apart ? -1 : q, CA_UPD_PARK, -1, L.f_g[j], 0, apart ? 1 : 0);
    step(L.pa[q], CA_X, OP_DX, L.f_g[j], 0, 1);
    step(L.pb[q], CA_PARKED, OP_DY, L.f_g[j], 1);
  }
  if (L.model == SW_MODEL_SW) {
    task(CT_H, 0);
    step(L.p_hu, CA_PARK, -1, -1);
    if (split) step(L.p_hv, CA_KEEP, -1, -1, 1);
    step(split ? -1 : L.p_hv, CA_UPD, -1, L.f_h, 1, 1);
    step(L.i_h, CA_X, OP_ID, L.f_h, 1);
  }
}

// ---------------------------------------------------------------------------
// Algorithmic bytes of one launch of each stepping kernel for one run: the
// distinct input elements it must read and the output elements it must write
// (box modes NY*KX, mixed rows N*KX, physical N*N), not counting L2 hits or
// padding.
struct KBytes {
  double col_inv, row_inv, row_prod, col_stage[4];
};

static KBytes kernel_bytes(const sw_handle* h, const Layout& L) {
  const Geom& g = h->g;
  const double cs = 2.0 * h->tsz, ts = (double)h->tsz;
  const double MB = (double)g.NY * g.KX, MI = (double)g.N * g.KX, NP = (double)g.np;
  KBytes b;
  bool seen[MAXF] = {};
  int nsrc = 0;
  for (int i = 0; i < L.ni; ++i) {
    if (!seen[L.i_src[i]]) { seen[L.i_src[i]] = true; ++nsrc; }
    if (L.i_src2[i] >= 0 && !seen[L.i_src2[i]]) { seen[L.i_src2[i]] = true; ++nsrc; }
  }
  b.col_inv = nsrc * MB * cs + L.ni * MI * cs;
  // row inverse pass: u, v, h, zeta (and xi, q) rows to physical planes, for
  // the runs whose row pass does not form them itself
  const int base = L.strategy == 2 ? 6 : 4;
  const bool fused = h->fp32 ? row_prod_fused<float>(g.N, L) : row_prod_fused<double>(g.N, L);
  b.row_inv = fused ? 0.0 : base * MI * cs + (base + (L.strategy == 2 && L.has_q)) * NP * ts;
  // row pass: mixed rows (or gradients, and the base planes) in, products
  // out; Strategy 2 also gathers q (the other gathered planes are base planes)
  double rp = L.np * MI * cs + (fused ? L.ni * MI * cs : (L.ni - base) * MI * cs + base * NP * ts);
  if (L.strategy == 2) {
    bool gq = false;
    for (int p = 0; p < L.np; ++p)
      if (L.pk[p] == PK_GBAR && L.pc[p] == PH_Q) gq = true;
    if (gq) rp += NP * ts;
  }
  b.row_prod = rp;
  int nk = 0, ne = 0;
  for (int f = 0; f < L.nf; ++f) {
    nk += L.fkahan[f];
    ne += L.frole[f] == R_E;
  }
  const double nf = L.nf, mixed = (L.np + (L.np > 0 ? L.ni : 0)) * MI * cs;
  // column stage: mixed products in, mixed fields out; y_n (not of the
  // Eulerian accumulators before the commit), the accumulator, the stage
  // inputs and outputs of u, v, h; integrating factors per class: E at every
  // stage, E^2 as hi + lo at the commit
  const bool rk4 = h->p.stepper == SW_STEP_RK4;
  const int last = stage_count(h->p.stepper) - 1;
  for (int st = 0; st < 4; ++st) {
    if (st >= last)
      b.col_stage[st] = mixed + (2 * nf + nf + 3 + (h->fp32 ? 2 * nk : 0)) * MB * cs + 4 * MB * ts;
    else
      b.col_stage[st] = mixed + ((nf - ne) + nf * (rk4 && st > 0 ? 2 : 1) + (st > 0 ? 3 : 0) + 3) * MB * cs + 2 * MB * ts;
  }
  return b;
}

// Optional per-launch event bracketing (sw_kernel_times).
struct Prof {
  enum { MAXEV = 64 };
  cudaEvent_t ev[2 * MAXEV];
  int cls[MAXEV];
  double bytes[MAXEV];
  int n = 0;
};

// ---------------------------------------------------------------------------
// Batch executor: the device table of run descriptors, per-kernel block
// prefix sums and the captured step graphs for a set of handles.
static const int GRAPH_STEPS = 8;
static const long long SMS = 152;  // of a GB300
// warps in the row pass below which its products are split over blocks
static const long long ROW_WARPS = 8 * SMS;
// Column-stage blocks up to which blocks are split in quarters (the two blocks
// an SM holds; a step of one Strategy-1 run, halves -> quarters: FP64 64^2 157 -> 141
// us, 128^2 190 -> 172, 16^2 dynamics 136 -> 123; FP32 128^2 64 -> 61) and in halves
// (beyond one wave: half of 456 blocks still end sooner than the whole ones: FP64 two
// 128^2 runs, 384 blocks, whole 297 -> 226 us, 256^2 Strategy 2, 352 blocks, 451 -> 427;
// FP32 256^2 both strategies, 352 blocks, 122 -> 117).
static const long long QUAD_BLOCKS = 2 * SMS;
static const long long DUAL_BLOCKS = 3 * SMS;
static const int SW_K_OF_KT[KT_COUNT] = {SW_K_ROW_INV, SW_K_ROW_PROD, SW_K_COL_STAGE, SW_K_UPDATE};

struct BatchExec {
  std::vector<sw_handle*> members;
  std::vector<uint64_t> versions;
  bool fp32 = false;
  cudaStream_t stream = nullptr;
  cudaStream_t cap = nullptr;  // private stream used only for graph capture
  int nruns = 0;
  void* d_table = nullptr;  // RunDesc<T>[nruns] then int start[KT_COUNT][nruns+1]
  size_t table_bytes = 0;
  int* d_start = nullptr;
  std::vector<int> start;
  int threads[KT_COUNT] = {};
  size_t smem[KT_COUNT] = {};
  double bytes[KT_COUNT][4] = {};
  double start_bytes = 0.0;  // of the transform-only launch (0: not needed)
  cudaGraphExec_t g1 = nullptr, gm = nullptr, gf = nullptr;  // 1 step, GRAPH_STEPS steps, the final step
  int64_t kernels_per_step = 0;
  int64_t launches = 0;
  int64_t replayed = 0;  // kernels of the last replay
  bool built = false;
  int nstages = 4;  // stage passes per step of the members' (common) stepper
  int stepper = SW_STEP_RK4;
  int parts = 1;  // parts that column-stage blocks are split into
  bool warp = false;  // every member's N <= 256: row kernels without named barriers
  std::string err;
};

static void batch_drop_graphs(BatchExec* b) {
  if (b->g1) cudaGraphExecDestroy(b->g1);
  if (b->gm) cudaGraphExecDestroy(b->gm);
  if (b->gf) cudaGraphExecDestroy(b->gf);
  b->g1 = b->gm = b->gf = nullptr;
}

static void batch_free(BatchExec* b) {
  if (!b) return;
  batch_drop_graphs(b);
  if (b->cap) cudaStreamDestroy(b->cap);
  if (b->d_table) cudaFree(b->d_table);
  delete b;
}

template <typename T>
static void fill_desc(sw_handle* h, RunDesc<T>& d, int points, int ppb, int lC, int parts, bool team) {
  std::memset(&d, 0, sizeof(d));
  const Geom& g = h->g;
  d.g = g;
  d.L = h->L;
  build_tasks(d.L, parts);
  d.c = StepConsts{h->p.dt, h->p.f0, h->p.c2, h->p.adv_x, h->p.adv_y, h->p.stepper, 0};
  d.cdt = (T)h->p.dt;
  d.cf0 = (T)h->p.f0;
  d.cc2 = (T)h->p.c2;
  d.cadvx = (T)h->p.adv_x;
  d.cadvy = (T)h->p.adv_y;
  d.cci = h->p.stepper == SW_STEP_RK4 ? d.cdt / (T)6 : (h->p.stepper == SW_STEP_HEUN ? d.cdt / (T)2 : (T)1);
  d.y = (cplx<T>*)h->y;
  d.ysa = (cplx<T>*)h->ys;
  d.ysb = (cplx<T>*)h->ys2;
  d.acc = (cplx<T>*)h->acc;
  d.comp = h->fp32 ? (cplx<T>*)h->comp : nullptr;
  d.mix = (cplx<T>*)h->mix;
  d.pmix = (cplx<T>*)h->pmix;
  d.phys = (T*)h->phys;
  d.ef = (const T*)h->ef;
  d.tw = (const twid<T>*)h->tw;
  d.ctr = h->ctr;
  d.ticket = h->ticket;
  d.lC = lC;
  const Layout& L = h->L;
  d.Bp = row_block_pairs(g.N, points);
  d.ppb = ppb < L.np || L.np == 0 ? ppb : L.np;
  d.Wp = 1;
  d.Bi = row_inv_pairs(g.N, points);
  const int ntile = g.KXP >> lC;
  const int chunks = L.np > 0 ? (L.np + d.ppb - 1) / d.ppb : 0;
  for (int q = 0; q < L.np; ++q) {
    // base fields product q is formed from
    const int k = L.pk[q], u = 1 << PH_U, v = 1 << PH_V, e = 1 << PH_H, z = 1 << PH_Z;
    d.umask[q / d.ppb] |= k == PK_ZV ? z | v : k == PK_ZU ? z | u : k == PK_KE ? u | v : k == PK_HU ? e | u
                        : k == PK_HV ? e | v : k == PK_Q ? z | e : (k == PK_ADV && L.model != 1) ? u | v : 0;
  }
  d.fused = row_prod_fused<T>(g.N, L) ? 1 : 0;
  d.gath = row_prod_gath<T>(g.N, L) && d.ppb >= L.np ? 1 : 0;
  d.team = team ? 1 : 0;
  // (a launch below a wave of blocks is as long as its longest block: 256^2
  // 103 -> 101 us a step; above, fewer blocks of more work: 2048^2 67 us against 74)
  d.hzsep = !team && !L.has_q && g.N <= 256 ? 1 : 0;
  d.nb[KT_ROW_INV] =
      L.np > 0 && !d.fused ? ((L.strategy == 2 ? 5 : 3) + d.hzsep) * row_blocks(g.N, d.Bi) : 0;
  d.nb[KT_ROW_PROD] = row_blocks(g.N, d.Bp) * chunks;
  d.nb[KT_COL_STAGE] = L.np > 0 ? ntile * d.L.nct : 0;
  d.nb[KT_KIN] = L.np > 0 ? 0 : (int)((g.ms + kin_modes(g.N) - 1) / kin_modes(g.N));
}

// Build (or rebuild) the descriptor table of a batch from its members.
template <typename T>
static int batch_build_t(BatchExec* b) {
  const int n = (int)b->members.size();
  std::vector<RunDesc<T>> descs(n);
  for (int k = 0; k < KT_COUNT; ++k) {
    b->threads[k] = 0;
    b->smem[k] = 0;
    for (int st = 0; st < 4; ++st) b->bytes[k][st] = 0.0;
  }
  b->start_bytes = 0.0;
  b->start.assign((size_t)KT_COUNT * (n + 1), 0);
  const size_t cs = sizeof(cplx<T>);
  for (int r = 1; r < n; ++r)
    if (b->members[r]->p.stepper != b->members[0]->p.stepper) {
      b->err = "batch members need the same stepper";
      return SW_EINVAL;
    }
  b->stepper = n > 0 ? b->members[0]->p.stepper : SW_STEP_RK4;
  b->nstages = stage_count(b->stepper);
  // members with transforms need one grid size, or sizes from 64 to 512 (equal
  // block shapes); members without (kinematic dynamics) have no such need
  {
    int lo = 0, hi = 0;
    for (int r = 0; r < n; ++r) {
      const int N = b->members[r]->g.N;
      if (b->members[r]->L.np == 0) continue;
      lo = lo ? std::min(lo, N) : N;
      hi = std::max(hi, N);
    }
    if (lo != hi && (lo < 64 || hi > 512)) {
      b->err = "batch members need equal block shapes (grid sizes 64..512, or one grid size)";
      return SW_EINVAL;
    }
  }
  b->warp = true;
  for (int r = 0; r < n; ++r) b->warp = b->warp && (b->members[r]->g.N <= 256 || b->members[r]->L.np == 0);
  // row pass: products per block (automatic: all of them, unless that leaves
  // the GPU short of warps, see below) and groups per row pair, the largest
  // number every member allows (the batch's row-pass blocks all have
  // Bp * Wp * N/8 threads)
  int points = 0;
  for (int r = 0; r < n; ++r)
    if (b->members[r]->L.np > 0) points = std::max(points, std::max(b->members[r]->points, b->members[r]->g.N));
  // (fewer row pairs where a block's arrays would not fit)
  auto fits = [&](int pts) {
    for (int r = 0; r < n; ++r) {
      const sw_handle* h = b->members[r];
      if (h->L.np > 0 && row_prod_smem<T>(h->g.N, row_block_pairs(h->g.N, pts), 1, h->L) > (size_t)200 * 1024) {
        if (pts > 256) return false;
      }
    }
    return true;
  };
  while (!fits(points)) {
    bool half = true;
    for (int r = 0; r < n; ++r) half = half && (b->members[r]->L.np == 0 || points / 2 >= b->members[r]->g.N);
    if (!half) break;
    points /= 2;
  }
  long long row_blks = 0;
  for (int r = 0; r < n; ++r) {
    const int N = b->members[r]->g.N;
    if (b->members[r]->L.np > 0) row_blks += row_blocks(N, row_block_pairs(N, points));
  }
  auto groups = [&](const sw_handle* h, int npb) {
    return row_prod_groups<T>(h->g.N, row_block_pairs(h->g.N, points), npb < h->L.np ? npb : h->L.np, h->L,
                              row_blks <= SMS);
  };
  int W = 1 << 20;
  long long warps = 0;
  for (int r = 0; r < n; ++r) {
    const sw_handle* h = b->members[r];
    if (h->L.np > 0) W = std::min(W, groups(h, h->ppb > 0 ? h->ppb : MAXP));
  }
  if (W > MAXP) W = 1;
  for (int r = 0; r < n; ++r) {
    const sw_handle* h = b->members[r];
    if (h->L.np > 0) warps += std::max<long long>(1, (long long)W * (h->g.N / 2) * (h->g.N / 8) / 32);
  }
  // fewer warps than ROW_WARPS (8 per SM): the products are split over
  // blocks, each transforming the base fields its products need.  Not where
  // several groups per row pair share them, in FP32: a split gives up the shared
  // base fields and gather (256^2, split -> not: dynamics 63 -> 51 us a step, Strategy
  // 2 of one field 104 -> 98; FP64, bound by issue, the other way round: Strategy 1 of
  // four 302 against 328)
  const int chunks =
      warps == 0 || (W > 1 && sizeof(T) == 4) ? 1 : (int)std::min<long long>(MAXP, (ROW_WARPS + warps - 1) / warps);
  auto products = [&](const sw_handle* h) {
    return h->ppb != 0 ? h->ppb : std::max(1, (h->L.np + chunks - 1) / chunks);
  };
  bool team = warps > 0;
  long long team_blocks = 0;
  for (int r = 0; r < n; ++r) {
    const sw_handle* h = b->members[r];
    if (h->L.np == 0) continue;
    team = team && row_team<T>(h->g.N, points, products(h));
    team_blocks += (long long)row_blocks(h->g.N, row_block_pairs(h->g.N, points)) * h->L.np;
  }
  team = team && team_blocks <= SMS * row_team_blocks<T>();
  // column tiles: the narrowest that still move whole 32-byte sectors (4 FP32
  // or 2 FP64 columns of the largest grid, 1 at 2048^2 in FP64), at least a
  // warp per block; the same points per block for every member.  Narrow tiles
  // spread a grid over more SMs (column stage at 64^2 in FP64: 62 us with 2048
  // points per block, 42 us so)
  int P = 256;
  for (int r = 0; r < n; ++r)
    if (b->members[r]->L.np > 0) P = std::max(P, b->members[r]->g.N * (sizeof(T) == 4 ? 4 : 2));
  if (sizeof(T) == 8) P = std::min(P, 2048);
  // split column blocks (see ColShape)
  long long col_blocks = 0;
  for (int r = 0; r < n; ++r) {
    const Layout& L = b->members[r]->L;
    if (L.np > 0) col_blocks += (long long)b->members[r]->g.KXP * b->members[r]->g.N / P * (L.nlm + (L.has_pos ? 2 : 0) + 2);
  }
  b->parts = P / 2 <= SPLIT_THREADS<T>() && col_blocks <= QUAD_BLOCKS ? 4
             : P / 4 <= SPLIT_THREADS<T>() && col_blocks <= DUAL_BLOCKS ? 2 : 1;
  for (int r = 0; r < n; ++r) {
    sw_handle* h = b->members[r];
    int lC = 0;
    while ((h->g.N << lC) < P && lC < h->lC) ++lC;
    fill_desc<T>(h, descs[r], points, products(h), lC, b->parts, team);
    descs[r].Wp = team ? 4 : W;
    const RunDesc<T>& d = descs[r];
    const int N = h->g.N;
    const int cthr = (N << lC) / 8;
    const size_t csm = ((size_t)col_buf_stride<T>(N, 1 << lC) << lC) * cs;
    const int sets = team ? 4 : 1;
    const int thr[KT_COUNT] = {sets * d.Bi * N / 8, d.Bp * d.Wp * N / 8, b->parts * cthr, 256};
    const size_t sm[KT_COUNT] = {(size_t)sets * 2 * d.Bi * row_stride<T>(N) * cs,
                                 row_prod_smem<T>(N, d.Bp, d.Wp, h->L, d.gath != 0),
                                 b->parts * csm + (size_t)6 * cthr * cs, 0};
    const KBytes kb = kernel_bytes(h, h->L);
    if (h->L.np > 0) b->start_bytes += kb.col_inv;
    const double by[KT_COUNT] = {kb.row_inv, kb.row_prod, 0.0, 0.0};
    for (int k = 0; k < KT_COUNT; ++k) {
      b->start[(size_t)k * (n + 1) + r + 1] = b->start[(size_t)k * (n + 1) + r] + d.nb[k];
      if (d.nb[k] == 0) continue;
      b->threads[k] = thr[k];
      if (sm[k] > b->smem[k]) b->smem[k] = sm[k];
      for (int st = 0; st < 4; ++st) b->bytes[k][st] += (k >= KT_COL_STAGE ? kb.col_stage[st] : by[k]);
    }
  }
  const size_t desc_bytes = (sizeof(RunDesc<T>) * n + 255) & ~(size_t)255;
  const size_t need = desc_bytes + sizeof(int) * b->start.size();
  if (need > b->table_bytes) {
    if (b->d_table) cudaFree(b->d_table);
    b->d_table = nullptr;
    cudaError_t e = cudaMalloc(&b->d_table, need);
    if (e != cudaSuccess) {
      cudaGetLastError();
      b->table_bytes = 0;
      b->err = std::string("cudaMalloc (batch table): ") + cudaGetErrorString(e);
      return SW_ENOMEM;
    }
    b->table_bytes = need;
  }
  b->d_start = (int*)((char*)b->d_table + desc_bytes);
  cudaError_t e = cudaMemcpyAsync(b->d_table, descs.data(), sizeof(RunDesc<T>) * n, cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(b->d_start, b->start.data(), sizeof(int) * b->start.size(), cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) {
    b->err = std::string("batch table upload: ") + cudaGetErrorString(e);
    return SW_ECUDA;
  }
  b->nruns = n;
  b->versions.resize(n);
  for (int r = 0; r < n; ++r) b->versions[r] = b->members[r]->version;
  batch_drop_graphs(b);
  b->built = true;
  return SW_OK;
}

static int batch_build(BatchExec* b) { return b->fp32 ? batch_build_t<float>(b) : batch_build_t<double>(b); }

static bool batch_stale(const BatchExec* b) {
  if (!b->built) return true;
  for (size_t r = 0; r < b->members.size(); ++r)
    if (b->versions[r] != b->members[r]->version) return true;
  return false;
}

#define LAUNCH(cls_, bytes_, ...)                                    \
  do {                                                               \
    if (pf) cudaEventRecord(pf->ev[2 * pf->n], s);                   \
    if ((e = (__VA_ARGS__)) != cudaSuccess) return e;                \
    if (pf) {                                                        \
      cudaEventRecord(pf->ev[2 * pf->n + 1], s);                     \
      pf->cls[pf->n] = (cls_);                                       \
      pf->bytes[pf->n] = (bytes_);                                   \
      pf->n++;                                                       \
    }                                                                \
    ++*nlaunch;                                                      \
  } while (0)

// One kernel kind over the batch (nothing if no member has blocks of it).
template <typename T>
static cudaError_t enqueue_kernel(BatchExec* b, int k, int stage, bool fin, bool pdl, cudaStream_t s, Prof* pf,
                                  int64_t* nlaunch) {
  const int n = b->nruns;
  const int total = b->start[(size_t)k * (n + 1) + n];
  cudaError_t e;
  if (total == 0) return cudaSuccess;
  LAUNCH(stage < 0 ? SW_K_COL_INV : SW_K_OF_KT[k], stage < 0 ? b->start_bytes : b->bytes[k][stage],
         launch_stage<T>(k, (const RunDesc<T>*)b->d_table, b->d_start + (size_t)k * (n + 1), n, total, b->threads[k],
                         b->smem[k], fin ? stage | STAGE_FINAL : stage, b->warp, b->parts, pdl, s));
  return cudaSuccess;
}

// Before the first step of a replay: the mixed fields of the state.  (The
// state may have been set, and the layout changed, since the last one.)
template <typename T>
static cudaError_t enqueue_batch_start(BatchExec* b, cudaStream_t s, Prof* pf, int64_t* nlaunch) {
  if (b->start_bytes == 0.0) return cudaSuccess;  // no products: nothing reads the mixed fields
  return enqueue_kernel<T>(b, KT_COL_STAGE, -1, false, false, s, pf, nlaunch);
}

// One step of every member of the batch; leaves the mixed fields of the new
// state for the next one (not after the final step of a replay).
template <typename T>
static cudaError_t enqueue_batch_step(BatchExec* b, bool final_step, cudaStream_t s, Prof* pf, int64_t* nlaunch) {
  static const int order[] = {KT_ROW_INV, KT_ROW_PROD, KT_COL_STAGE, KT_KIN};
  for (int stage = 0; stage < b->nstages; ++stage) {
    // forward Euler's second pass only commits
    const bool commit_only = b->stepper == SW_STEP_EULER && stage == 1;
    for (int k : order) {
      if (commit_only && k != KT_COL_STAGE && k != KT_KIN) continue;
      const bool fin = final_step && k == KT_COL_STAGE && stage == b->nstages - 1;
      const cudaError_t e = enqueue_kernel<T>(b, k, stage, fin, pf == nullptr, s, pf, nlaunch);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

// Capture `steps` steps into an executable graph (`final_step`: the last of
// them ends a replay).  Capture runs on a
// private stream (the caller's stream may be the legacy default stream, which
// cannot be captured); the graphs are launched on the batch's stream.
static int batch_capture(BatchExec* b, int steps, bool final_step, cudaGraphExec_t* out) {
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaSuccess;
  if (!b->cap && (e = cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking)) != cudaSuccess) {
    b->err = std::string("cudaStreamCreate: ") + cudaGetErrorString(e);
    return SW_ECUDA;
  }
  if ((e = cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal)) != cudaSuccess) {
    b->err = std::string("cudaStreamBeginCapture: ") + cudaGetErrorString(e);
    return SW_ECUDA;
  }
  int64_t nl = 0;
  for (int i = 0; i < steps && e == cudaSuccess; ++i)
    e = b->fp32 ? enqueue_batch_step<float>(b, final_step, b->cap, nullptr, &nl)
                : enqueue_batch_step<double>(b, final_step, b->cap, nullptr, &nl);
  cudaError_t e2 = cudaStreamEndCapture(b->cap, &graph);
  if (e != cudaSuccess || e2 != cudaSuccess) {
    if (graph) cudaGraphDestroy(graph);
    b->err = std::string("step capture: ") + cudaGetErrorString(e != cudaSuccess ? e : e2);
    return SW_ECUDA;
  }
  e = cudaGraphInstantiate(out, graph, 0);
  cudaGraphDestroy(graph);
  if (e == cudaSuccess && (e = cudaGraphUpload(*out, b->stream)) != cudaSuccess)  // not at the first replay
    cudaGraphExecDestroy(*out);
  if (e != cudaSuccess) {
    *out = nullptr;
    b->err = std::string("cudaGraphInstantiate: ") + cudaGetErrorString(e);
    return SW_ECUDA;
  }
  b->kernels_per_step = nl / steps;
  return SW_OK;
}

static int batch_ready(BatchExec* b) {
  if (batch_stale(b)) {
    int rc = batch_build(b);
    if (rc) return rc;
  }
  if (!b->g1) {
    int rc = batch_capture(b, 1, false, &b->g1);
    if (rc == SW_OK) rc = batch_capture(b, 1, true, &b->gf);
    if (rc == SW_OK) rc = batch_capture(b, GRAPH_STEPS, false, &b->gm);
    if (rc != SW_OK) {
      batch_drop_graphs(b);
      return rc;
    }
  }
  return SW_OK;
}

// Replay n steps of the batch (no bookkeeping on the members).
static int batch_replay(BatchExec* b, int64_t n) {
  int rc = batch_ready(b);
  if (rc) return rc;
  int64_t nl = 0;
  cudaError_t e = b->fp32 ? enqueue_batch_start<float>(b, b->stream, nullptr, &nl)
                          : enqueue_batch_start<double>(b, b->stream, nullptr, &nl);
  int64_t i = 0;
  for (; e == cudaSuccess && i + GRAPH_STEPS < n; i += GRAPH_STEPS) e = cudaGraphLaunch(b->gm, b->stream);
  for (; e == cudaSuccess && i < n; ++i) e = cudaGraphLaunch(i + 1 < n ? b->g1 : b->gf, b->stream);
  if (e != cudaSuccess) {
    b->err = std::string("cudaGraphLaunch: ") + cudaGetErrorString(e);
    return SW_ECUDA;
  }
  b->replayed = n * b->kernels_per_step + nl;
  b->launches += b->replayed;
  return SW_OK;
}

static int run_steps(sw_handle* h, int64_t n) {
  if (n <= 0) return SW_OK;
  int rc = batch_replay(h->self, n);
  if (rc) return fail(h, rc, h->self->err);
  h->steps_total += n;
  h->launches += h->self->replayed;
  return SW_OK;
}

static void set_layout(sw_handle* h, const Layout& L) {
  h->L = L;
  ++h->version;
}

// ---------------------------------------------------------------------------
// FP64 transforms around the stepping.

// Physical FP64 fields (N*N each, in h->out64[slot..]) from up to two
// spectral fields of the state: value = (y - comp)*scale, plus ax*x + ay*y.
struct OutSpec {
  int field;  // evolved-field index (-1: none)
  double scale, ax, ay;
  int slot;   // output slot in out64
  double cst; // constant added (1 for the depth h = 1 + eta)
  int field2 = -1;  // >= 0: the curl i kx field2 - i ky field
};

template <typename T>
static int phys_outputs_t(sw_handle* h, const OutSpec* os, int n) {
  for (int i = 0; i < n; i += IO_MAX) {
    OutArgs<T> a;
    std::memset(&a, 0, sizeof(a));
    a.y = (const cplx<T>*)h->y;
    a.comp = h->fp32 ? (const cplx<T>*)h->comp : nullptr;
    a.mix = h->mix64;
    a.phys = h->out64;
    a.tw = h->tw64;
    a.g = h->g;
    a.n = n - i < IO_MAX ? n - i : IO_MAX;
    for (int q = 0; q < a.n; ++q) {
      const OutSpec& o = os[i + q];
      a.field[q] = o.field;
      a.field2[q] = o.field2;
      a.slot[q] = o.slot;
      a.scale[q] = o.scale;
      a.ax[q] = o.ax;
      a.ay[q] = o.ay;
      a.cst[q] = o.cst;
    }
    CK(h, launch_out<T>(a, h->stream));
    h->launches += 2;
  }
  return SW_OK;
}
static int phys_outputs(sw_handle* h, const OutSpec* os, int n) {
  return h->fp32 ? phys_outputs_t<float>(h, os, n) : phys_outputs_t<double>(h, os, n);
}

// Load a physical FP64 initial condition (already in out64[0..2]) into the
// dynamics fields of the state.
template <typename T>
static int load_ic_t(sw_handle* h) {
  InArgs<T> a;
  std::memset(&a, 0, sizeof(a));
  a.phys = h->out64;
  a.mix = h->mix64;
  a.y = (cplx<T>*)h->y;
  a.tw = h->tw64;
  a.g = h->g;
  a.n = 3;
  for (int i = 0; i < 3; ++i) a.slot[i] = a.field[i] = i;
  // the state holds the depth perturbation eta = h - 1 (mean depth 1 removed
  // from the k = 0 mode), which keeps its relative precision in FP32; the
  // two-dimensional Euler model holds the vorticity there and derives u, v
  const bool e2 = h->p.model == SW_MODEL_EULER2D;
  if (!e2) a.mean[2] = -1.0;
  CK(h, launch_in<T>(a, h->stream));
  if (e2) CK(h, launch_velocity_from_vorticity<T>((cplx<T>*)h->y, h->g, h->L.f_u, h->L.f_v, h->L.f_h, h->stream));
  h->launches += e2 ? 3 : 2;
  return SW_OK;
}
static int load_ic_from_out64(sw_handle* h) { return h->fp32 ? load_ic_t<float>(h) : load_ic_t<double>(h); }

static int copy_in_uvh(sw_handle* h, const double* uvh, int on_device) {
  const size_t bytes = (size_t)3 * h->g.np * sizeof(double);
  CK(h, cudaMemcpyAsync(h->out64, uvh, bytes, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                        h->stream));
  return load_ic_from_out64(h);
}

// ---------------------------------------------------------------------------
static bool is_pow2(int n) { return n > 0 && (n & (n - 1)) == 0; }

static int validate(const sw_params* p, std::string& why) {
  if (!p) { why = "params is NULL"; return SW_EINVAL; }
  if (!is_pow2(p->N) || p->N < 16 || p->N > 2048) { why = "N must be a power of two in [16, 2048]"; return SW_EINVAL; }
  if (p->precision != SW_PREC_FP64 && p->precision != SW_PREC_FP32) { why = "precision must be SW_PREC_FP64 or SW_PREC_FP32"; return SW_EINVAL; }
  if (p->model != SW_MODEL_SW && p->model != SW_MODEL_KINEMATIC && p->model != SW_MODEL_EULER2D) { why = "model must be SW_MODEL_SW, SW_MODEL_KINEMATIC or SW_MODEL_EULER2D"; return SW_EINVAL; }
  if (p->reserved != 0) { why = "reserved must be 0"; return SW_EINVAL; }
  if (p->stepper < SW_STEP_RK4 || p->stepper > SW_STEP_EULER) { why = "stepper must be SW_STEP_RK4, SW_STEP_HEUN or SW_STEP_EULER"; return SW_EINVAL; }
  if (p->visc != SW_VISC_HYPER8 && p->visc != SW_VISC_LAPLACE) { why = "visc must be SW_VISC_HYPER8 or SW_VISC_LAPLACE"; return SW_EINVAL; }
  if (!(p->dt > 0.0) || !std::isfinite(p->dt)) { why = "dt must be finite and > 0"; return SW_EINVAL; }
  if (!std::isfinite(p->f0) || !std::isfinite(p->adv_x) || !std::isfinite(p->adv_y)) { why = "f0 and adv must be finite"; return SW_EINVAL; }
  if (!(p->c2 >= 0.0) || !std::isfinite(p->c2)) { why = "c2 must be finite and >= 0"; return SW_EINVAL; }
  if (!(p->nu8 >= 0.0) || !(p->lm_nu8 >= 0.0) || !std::isfinite(p->nu8) || !std::isfinite(p->lm_nu8)) { why = "nu8, lm_nu8 must be finite and >= 0"; return SW_EINVAL; }
  return SW_OK;
}

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

static const int DIAG_BLOCKS = 1024;

// Grid geometry: cutoff K, the most columns 2^lC a column tile may have (2048/N, at
// most 32, so that grids of 64 to 512 can have tiles of equal points in a batch;
// in FP32 at least 4, which move whole 32-byte sectors; four FP64 columns of 2048
// points would not fit in shared memory; a launch's own tiles: batch_build_t) and the
// padded column count KXP (a multiple of 2^lC and of 4).
static void plan_geometry(int N, size_t tsz, Geom& g, int& lC) {
  g.N = N;
  g.log2N = 0;
  while ((1 << g.log2N) < g.N) ++g.log2N;
  g.K = (g.N - 1) / 3;
  g.KX = g.K + 1;
  lC = 0;
  while ((1 << lC) * g.N < 2048 && lC < 5) ++lC;
  if (tsz == 4 && lC < 2) lC = 2;
  const int C = 1 << lC;
  const int pad = C > 4 ? C : 4;
  g.KXP = (g.KX + pad - 1) / pad * pad;
  g.NY = 2 * g.K + 1;
  g.ms = (long long)g.NY * g.KXP;
  g.mi = (long long)g.N * g.KXP;
  g.np = (long long)g.N * g.N;
}

// Offsets of the handle's device arena (256-byte aligned slices).
struct ArenaPlan {
  size_t o[18];
  size_t total;
};

static ArenaPlan plan_arena(const Geom& g, size_t tsz) {
  ArenaPlan A;
  const size_t cs = 2 * tsz;
  const size_t sizes[18] = {
      MAXF * g.ms * cs, 3 * g.ms * cs, 3 * g.ms * cs, MAXF * g.ms * cs,        // y, ys, ys2, acc
      MAXF * g.ms * cs,                                                        // comp
      MAXI * g.mi * cs, MAXP * g.mi * cs,                                      // mix, pmix
      NPH * g.np * tsz, 6 * g.ms * tsz, g.N * cs,                              // phys, ef, tw
      g.N * sizeof(TwFx), g.ms * sizeof(double2),                              // tw64, spec64
      4 * g.mi * sizeof(double2), 12 * g.np * sizeof(double),                  // mix64, out64
      2 * DIAG_BLOCKS * sizeof(double), 4 * sizeof(double),                    // part, dres
      sizeof(long long), sizeof(unsigned)};                                    // ctr, ticket
  size_t off = 0;
  for (int i = 0; i < 18; ++i) {
    A.o[i] = off;
    off += align256(sizes[i]);
  }
  A.total = off;
  return A;
}

extern "C" int64_t sw_state_bytes(const sw_params* p) {
  std::string why;
  if (validate(p, why) != SW_OK) return 0;
  Geom g;
  int lC;
  const size_t tsz = p->precision == SW_PREC_FP32 ? 4 : 8;
  plan_geometry(p->N, tsz, g, lC);
  return (int64_t)plan_arena(g, tsz).total;
}

template <typename T>
static void host_tables(const sw_params& p, const Geom& g, void* ef_host, void* tw_host, TwFx* tw64_host) {
  T* ef = (T*)ef_host;
  static_assert(sizeof(twid<T>) == sizeof(cplx<T>), "twiddle table size");
  // per class (dynamics, mean fields): E = exp(-nu |k|^2p dt/2) for the
  // stage values, and E^2 as an unevaluated sum hi + lo for the commit
  // of y_{n+1} = E^2 y_n + ...: rounded to T alone, E^2 would move every
  // damped mode by up to half an ulp of T per step, an error that grows
  // linearly with the steps of an interval (in FP32 about 4e-5 after
  // 1219 steps at 64^2); hi + lo carries it to about twice T's digits.
  // In the order of the spectral layout; ky and -ky share their values.
  const double nus[2] = {p.nu8, p.lm_nu8};
  const int classes = p.nu8 == p.lm_nu8 ? 1 : 2;
  for (int c = 0; c < classes; ++c)
    for (int kx0 = 0; kx0 < g.KXP; kx0 += spec_tile<T>())
      for (int ky = 0; ky <= g.K; ++ky)
        for (int kx = kx0; kx < kx0 + spec_tile<T>(); ++kx) {
          const double k2 = (double)kx * kx + (double)ky * ky;
          const double k8 = p.visc == SW_VISC_LAPLACE ? k2 : k2 * k2 * k2 * k2;  // |k|^2p
          const double E = std::exp(-nus[c] * k8 * p.dt * 0.5);
          const double E2 = E * E;
          const T hi = (T)E2, lo = (T)(E2 - (double)hi);
          for (int sg = 0; sg < 2; ++sg) {
            const long long m = spec_index<T>(g.K + (sg ? -ky : ky), kx, g.NY);
            ef[(3 * c) * g.ms + m] = (T)E;
            ef[(3 * c + 1) * g.ms + m] = hi;
            ef[(3 * c + 2) * g.ms + m] = lo;
          }
        }
  if (classes == 1) std::memcpy(ef + 3 * g.ms, ef, 3 * g.ms * sizeof(T));
  fft_twiddle_table_fx(g.log2N, tw64_host);
  if (sizeof(T) == 8) {
    std::memcpy(tw_host, tw64_host, g.N * sizeof(TwFx));
  } else {
    std::vector<double> re(g.N, 1.0), im(g.N, 0.0);
    fft_twiddle_table(g.log2N, re.data(), im.data());
    for (int t = 0; t < g.N; ++t) ((float2*)tw_host)[t] = make_float2((float)re[t], (float)im[t]);
  }
}

extern "C" int sw_create(const sw_params* p, const double* ic_uvh, int ic_on_device, void* stream,
                         sw_handle** out) {
  g_create_error.clear();
  if (!out) return fail(nullptr, SW_EINVAL, "out is NULL");
  *out = nullptr;
  std::string why;
  int rc = validate(p, why);
  if (rc) return fail(nullptr, rc, why);
  if (!ic_uvh) return fail(nullptr, SW_EINVAL, "ic_uvh is NULL");
  static bool prepared = false;
  if (!prepared) {
    cudaError_t e = prepare_kernels_f32();
    if (e == cudaSuccess) e = prepare_kernels_f64();
    if (e != cudaSuccess) return fail(nullptr, SW_ECUDA, std::string("kernel set-up: ") + cudaGetErrorString(e));
    prepared = true;
  }
  sw_handle* h = new (std::nothrow) sw_handle();
  if (!h) return fail(nullptr, SW_ENOMEM, "host allocation failed");
  h->p = *p;
  h->stream = (cudaStream_t)stream;
  h->fp32 = p->precision == SW_PREC_FP32;
  h->tsz = h->fp32 ? 4 : 8;
  Geom& g = h->g;
  plan_geometry(p->N, h->tsz, g, h->lC);
  const size_t cs = 2 * h->tsz;  // complex T
  h->diag_blocks = DIAG_BLOCKS;
  h->ppb = 0;  // automatic (batch_build_t)
  const ArenaPlan A = plan_arena(g, h->tsz);
  const size_t o_y = A.o[0], o_ys = A.o[1], o_ys2 = A.o[2], o_acc = A.o[3], o_comp = A.o[4];
  const size_t o_mix = A.o[5], o_pmix = A.o[6], o_phys = A.o[7], o_ef = A.o[8], o_tw = A.o[9];
  const size_t o_tw64 = A.o[10], o_spec64 = A.o[11], o_mix64 = A.o[12], o_out64 = A.o[13];
  const size_t o_part = A.o[14], o_dres = A.o[15], o_ctr = A.o[16], o_ticket = A.o[17];
  const size_t off = A.total;
  h->arena_bytes = off;
  cudaError_t e = cudaMalloc(&h->arena, h->arena_bytes);
  if (e != cudaSuccess) {
    delete h;
    cudaGetLastError();
    return fail(nullptr, SW_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
  }
  char* base = (char*)h->arena;
  h->y = base + o_y; h->ys = base + o_ys; h->ys2 = base + o_ys2; h->acc = base + o_acc; h->comp = base + o_comp;
  h->mix = base + o_mix; h->pmix = base + o_pmix; h->phys = base + o_phys; h->ef = base + o_ef;
  h->tw = base + o_tw; h->tw64 = (TwFx*)(base + o_tw64); h->spec64 = (double2*)(base + o_spec64);
  h->mix64 = (double2*)(base + o_mix64); h->out64 = (double*)(base + o_out64);
  h->part = (double*)(base + o_part); h->dres = (double*)(base + o_dres);
  h->ctr = (long long*)(base + o_ctr); h->ticket = (unsigned*)(base + o_ticket);
  // tables
  const size_t ef_bytes = 6 * g.ms * h->tsz, tw_bytes = g.N * cs;
  char* hbuf = (char*)std::malloc(ef_bytes + tw_bytes + g.N * sizeof(TwFx));
  if (!hbuf) {
    cudaFree(h->arena);
    delete h;
    return fail(nullptr, SW_ENOMEM, "host allocation failed");
  }
  if (h->fp32) host_tables<float>(*p, g, hbuf, hbuf + ef_bytes, (TwFx*)(hbuf + ef_bytes + tw_bytes));
  else host_tables<double>(*p, g, hbuf, hbuf + ef_bytes, (TwFx*)(hbuf + ef_bytes + tw_bytes));
  rc = SW_OK;
  do {
    if ((e = cudaMemsetAsync(h->arena, 0, h->arena_bytes, h->stream)) != cudaSuccess) break;
    if ((e = cudaMemcpyAsync(h->ef, hbuf, ef_bytes, cudaMemcpyHostToDevice, h->stream)) != cudaSuccess) break;
    if ((e = cudaMemcpyAsync(h->tw, hbuf + ef_bytes, tw_bytes, cudaMemcpyHostToDevice, h->stream)) != cudaSuccess) break;
    if ((e = cudaMemcpyAsync(h->tw64, hbuf + ef_bytes + tw_bytes, g.N * sizeof(TwFx), cudaMemcpyHostToDevice,
                             h->stream)) != cudaSuccess) break;
    if ((e = cudaStreamSynchronize(h->stream)) != cudaSuccess) break;
  } while (0);
  std::free(hbuf);
  if (e != cudaSuccess) {
    std::string m = std::string("device set-up: ") + cudaGetErrorString(e);
    cudaFree(h->arena);
    delete h;
    return fail(nullptr, SW_ECUDA, m);
  }
  h->L = build_layout(*p, 0, 0, 0);
  h->self = new (std::nothrow) BatchExec();
  if (!h->self) {
    cudaFree(h->arena);
    delete h;
    return fail(nullptr, SW_ENOMEM, "host allocation failed");
  }
  h->self->members.push_back(h);
  h->self->fp32 = h->fp32;
  h->self->stream = h->stream;
  rc = copy_in_uvh(h, ic_uvh, ic_on_device);
  if (rc == SW_OK) {
    e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) rc = fail_cuda(h, "initial transform", e);
  }
  if (rc != SW_OK) {
    std::string m = h->err;
    batch_free(h->self);
    cudaFree(h->arena);
    delete h;
    return fail(nullptr, rc, m);
  }
  *out = h;
  return SW_OK;
}

extern "C" void sw_destroy(sw_handle* h) {
  if (!h) return;
  cudaStreamSynchronize(h->stream);
  batch_free(h->self);
  if (h->arena) cudaFree(h->arena);
  delete h;
}

extern "C" int sw_step(sw_handle* h, int64_t nsteps) {
  if (!h) return SW_EINVAL;
  h->err.clear();
  if (nsteps < 0) return fail(h, SW_EINVAL, "nsteps < 0");
  if (h->lm_open) return fail(h, SW_EBUSY, "an averaging interval is open");
  return run_steps(h, nsteps);
}

extern "C" int lmean_begin(sw_handle* h, const lm_params* lp) {
  if (!h) return SW_EINVAL;
  h->err.clear();
  if (!lp) return fail(h, SW_EINVAL, "lm_params is NULL");
  if (h->lm_open) return fail(h, SW_ESTATE, "an averaging interval is already open");
  if (lp->strategy != 1 && lp->strategy != 2) return fail(h, SW_EINVAL, "strategy must be 1 or 2");
  if (lp->scheme != LM_SCHEME_COUPLED && lp->scheme != LM_SCHEME_XI_FIRST)
    return fail(h, SW_EINVAL, "scheme must be LM_SCHEME_COUPLED or LM_SCHEME_XI_FIRST");
  if (lp->scheme == LM_SCHEME_XI_FIRST &&
      (lp->strategy != 2 || h->p.stepper != SW_STEP_EULER || (lp->n_steps & 1)))
    return fail(h, SW_EINVAL, "LM_SCHEME_XI_FIRST needs strategy 2, SW_STEP_EULER and an even n_steps");
  if (lp->n_steps < 1) return fail(h, SW_EINVAL, "n_steps must be >= 1");
  if (lp->fields & ~(LM_ZETA | LM_H | LM_U | LM_V | LM_Q | LM_POS))
    return fail(h, SW_EINVAL, "unknown bits in fields");
  const int scal = lp->fields & (LM_ZETA | LM_H | LM_U | LM_V | LM_Q);
  if (!scal && !(lp->fields & LM_POS)) return fail(h, SW_EINVAL, "no field selected");
  if (h->p.model == SW_MODEL_EULER2D && (lp->fields & (LM_H | LM_Q)))
    return fail(h, SW_EINVAL, "the two-dimensional Euler model averages zeta, u and v only");
  if (!scal && lp->eulerian) return fail(h, SW_EINVAL, "Eulerian means need a scalar field");
  Layout L = build_layout(h->p, lp->strategy, lp->fields, lp->eulerian, lp->scheme);
  const Geom& g = h->g;
  const size_t cs = 2 * h->tsz;
  // zero the mean fields, their compensation terms and the step counter
  CK(h, cudaMemsetAsync((char*)h->y + 3 * g.ms * cs, 0, (size_t)(MAXF - 3) * g.ms * cs, h->stream));
  CK(h, cudaMemsetAsync(h->comp, 0, (size_t)MAXF * g.ms * cs, h->stream));
  CK(h, cudaMemsetAsync(h->ctr, 0, sizeof(long long), h->stream));
  set_layout(h, L);
  h->lp = *lp;
  h->done = 0;
  h->lm_open = true;
  return SW_OK;
}

extern "C" int lmean_step(sw_handle* h, int64_t nsteps) {
  if (!h) return SW_EINVAL;
  h->err.clear();
  if (!h->lm_open) return fail(h, SW_ESTATE, "no averaging interval is open");
  if (nsteps < 0) return fail(h, SW_EINVAL, "nsteps < 0");
  if (nsteps > h->lp.n_steps - h->done) return fail(h, SW_ERANGE, "more steps than remain in the interval");
  int rc = run_steps(h, nsteps);
  if (rc == SW_OK) h->done += nsteps;
  return rc;
}

extern "C" int lmean_progress(sw_handle* h, int64_t* done, int64_t* remaining) {
  if (!h) return SW_EINVAL;
  if (done) *done = h->lm_open ? h->done : 0;
  if (remaining) *remaining = h->lm_open ? h->lp.n_steps - h->done : 0;
  return SW_OK;
}

static int copy_out(sw_handle* h, double* dst, int slot, int on_device) {
  if (!dst) return SW_OK;
  const size_t bytes = (size_t)h->g.np * sizeof(double);
  CK(h, cudaMemcpyAsync(dst, h->out64 + (size_t)slot * h->g.np, bytes,
                        on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, h->stream));
  return SW_OK;
}

extern "C" int lmean_end(sw_handle* h, const lm_result* out) {
  if (!h) return SW_EINVAL;
  h->err.clear();
  if (!h->lm_open) return fail(h, SW_ESTATE, "no averaging interval is open");
  if (h->done != h->lp.n_steps) return fail(h, SW_ESTATE, "interval not complete");
  if (!out) return fail(h, SW_EINVAL, "out is NULL");
  const Layout& L = h->L;
  const double T = (double)h->lp.n_steps * h->p.dt;
  double* lm_ptr[NLMF] = {out->zeta, out->h, out->u, out->v, out->q};
  double* e_ptr[NLMF] = {out->e_zeta, out->e_h, out->e_u, out->e_v, out->e_q};
  bool in_mask[NLMF] = {false, false, false, false, false};
  for (int j = 0; j < L.nlm; ++j) in_mask[L.lmf[j]] = true;
  for (int f = 0; f < NLMF; ++f) {
    if (lm_ptr[f] && !in_mask[f]) return fail(h, SW_EINVAL, "output requested for a field not averaged");
    if (e_ptr[f] && (!in_mask[f] || !L.eulerian)) return fail(h, SW_EINVAL, "Eulerian output not accumulated");
  }
  if ((out->pos_x || out->pos_y) && !L.has_pos) return fail(h, SW_EINVAL, "positions not computed");
  OutSpec os[12];
  double* dst[12];
  int n = 0;
  for (int j = 0; j < L.nlm; ++j)
    if (lm_ptr[L.lmf[j]]) {
      os[n] = OutSpec{L.f_g[j], 1.0 / T, 0.0, 0.0, n, L.lmf[j] == LMF_H ? 1.0 : 0.0};
      dst[n++] = lm_ptr[L.lmf[j]];
    }
  if (L.has_pos) {
    double* pp[2] = {out->pos_x, out->pos_y};
    for (int c = 0; c < 2; ++c)
      if (pp[c]) {
        // S1: Xi^{-1} = x - D/T;  S2: Xi = x + xi
        const double sc = L.strategy == 1 ? -1.0 / T : 1.0;
        os[n] = OutSpec{L.f_p[c], sc, c == 0 ? 1.0 : 0.0, c == 1 ? 1.0 : 0.0, n, 0.0};
        dst[n++] = pp[c];
      }
  }
  if (L.eulerian)
    for (int j = 0; j < L.nlm; ++j)
      if (e_ptr[L.lmf[j]]) {
        os[n] = OutSpec{L.f_e[j], 1.0 / T, 0.0, 0.0, n, L.lmf[j] == LMF_H ? 1.0 : 0.0};
        dst[n++] = e_ptr[L.lmf[j]];
      }
  int rc = phys_outputs(h, os, n);
  if (rc) return rc;
  for (int i = 0; i < n; ++i)
    if ((rc = copy_out(h, dst[i], i, out->on_device))) return rc;
  if (!out->on_device) CK(h, cudaStreamSynchronize(h->stream));
  h->lm_open = false;
  set_layout(h, build_layout(h->p, 0, 0, 0));
  return SW_OK;
}

extern "C" int sw_get_fields(sw_handle* h, double* uvh, int on_device) {
  if (!h) return SW_EINVAL;
  h->err.clear();
  if (!uvh) return fail(h, SW_EINVAL, "uvh is NULL");
  // third field: h = 1 + eta (zeta for the two-dimensional Euler model)
  const double c3 = h->p.model == SW_MODEL_EULER2D ? 0.0 : 1.0;
  OutSpec os[3] = {{h->L.f_u, 1.0, 0, 0, 0, 0.0}, {h->L.f_v, 1.0, 0, 0, 1, 0.0}, {h->L.f_h, 1.0, 0, 0, 2, c3}};
  // the dynamics fields carry no compensation term (it stays zero)
  int rc = phys_outputs(h, os, 3);
  if (rc) return rc;
  CK(h, cudaMemcpyAsync(uvh, h->out64, (size_t)3 * h->g.np * sizeof(double),
                        on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, h->stream));
  CK(h, cudaStreamSynchronize(h->stream));
  return SW_OK;
}

extern "C" int sw_set_fields(sw_handle* h, const double* uvh, int on_device) {
  if (!h) return SW_EINVAL;
  h->err.clear();
  if (!uvh) return fail(h, SW_EINVAL, "uvh is NULL");
  if (h->lm_open) return fail(h, SW_EBUSY, "an averaging interval is open");
  int rc = copy_in_uvh(h, uvh, on_device);
  if (rc) return rc;
  CK(h, cudaStreamSynchronize(h->stream));
  return SW_OK;
}

// Physical FP64 u, v, h, zeta of the current state in out64 slots 0..3
// (zeta by a spectral curl in FP64), on the handle's stream.
static int phys_uvhz(sw_handle* h) {
  const bool e2 = h->p.model == SW_MODEL_EULER2D;
  // (the dynamics fields carry no compensation term: it stays zero)
  OutSpec os[4] = {{h->L.f_u, 1.0, 0, 0, 0, 0.0}, {h->L.f_v, 1.0, 0, 0, 1, 0.0},
                   {h->L.f_h, 1.0, 0, 0, 2, e2 ? 0.0 : 1.0}, {h->L.f_u, 1.0, 0, 0, 3, 0.0, h->L.f_v}};
  // the evolved vorticity (with its mean) in both the h and the zeta slot
  if (e2) os[3] = OutSpec{h->L.f_h, 1.0, 0, 0, 3, 0.0};
  return phys_outputs(h, os, 4);
}

namespace lm {
// hooks for the semi-Lagrangian interval (gbla.cu)
int handle_info(sw_handle* h, HandleInfo* hi) {
  if (!h || !hi) return SW_EINVAL;
  hi->N = h->g.N;
  hi->dt = h->p.dt;
  hi->f0 = h->p.f0;
  hi->adv_x = h->p.adv_x;
  hi->adv_y = h->p.adv_y;
  hi->model = h->p.model;
  hi->lm_open = h->lm_open;
  hi->stream = h->stream;
  return SW_OK;
}
int handle_phys_uvhz(sw_handle* h, const double** out) {
  const int rc = phys_uvhz(h);
  if (rc) return rc;
  *out = h->out64;
  return SW_OK;
}
void handle_set_error(sw_handle* h, const std::string& msg) {
  if (h) h->err = msg;
}
}  // namespace lm

extern "C" int sw_diag(sw_handle* h, double out[3]) {
  if (!h) return SW_EINVAL;
  h->err.clear();
  if (!out) return fail(h, SW_EINVAL, "out is NULL");
  if (h->p.model == SW_MODEL_EULER2D) return fail(h, SW_EINVAL, "sw_diag has no two-dimensional Euler form");
  int rc = phys_uvhz(h);
  if (rc) return rc;
  const Geom& g = h->g;
  CK(h, launch_diag(h->out64, g.np, h->p.f0, h->p.c2, h->part, h->diag_blocks, h->dres, h->stream));
  h->launches += 2;  // (phys_uvhz counts its own)
  double res[4] = {0, 0, 0, 0};
  CK(h, cudaMemcpyAsync(res, h->dres, 3 * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  // mass: the k = 0 coefficient of h (row ky = 0, column kx = 0)
  const size_t cs = 2 * h->tsz;
  unsigned char m0[16];
  CK(h, cudaMemcpyAsync(m0, (char*)h->y +
                            ((size_t)h->L.f_h * g.ms + (h->fp32 ? spec_index<float>(g.K, 0, g.NY)
                                                                : spec_index<double>(g.K, 0, g.NY))) * cs, cs,
                        cudaMemcpyDeviceToHost, h->stream));
  CK(h, cudaStreamSynchronize(h->stream));
  // the state holds eta = h - 1
  out[0] = 1.0 + (h->fp32 ? (double)((float*)m0)[0] : ((double*)m0)[0]);
  out[1] = res[1];
  out[2] = res[2];
  return SW_OK;
}

// ---------------------------------------------------------------------------
// Checkpoint blob: header, then the evolved fields and their compensation.
struct BlobHeader {
  char magic[8];
  int32_t version, N, precision, model;
  double dt, f0, c2, nu8, lm_nu8, adv_x, adv_y;
  int32_t stepper, visc;
  int32_t lm_open, nf;
  lm_params lp;
  int64_t done, steps_total;
};

// The state's nf fields and compensation terms from (to_rows) or to rows
// [ky + K][kx], as blobs hold them, in the mixed fields' buffer, which the next
// replay fills anew; from rows, the step counter too.  (2 x 16 spectral fields
// of 2K + 1 < 2N/3 rows fit in its 24 fields of N rows.)
static_assert(2 * MAXF * 2 <= 3 * MAXI, "blob staging");
static int spec_rows(sw_handle* h, int nf, bool to_rows, long long done = 0) {
  if (h->fp32)
    CK(h, launch_spec_rows<float>((float2*)h->y, (float2*)h->comp, (float2*)h->mix, h->g, nf, to_rows, h->ctr, done,
                                  h->stream));
  else
    CK(h, launch_spec_rows<double>((double2*)h->y, (double2*)h->comp, (double2*)h->mix, h->g, nf, to_rows, h->ctr, done,
                                   h->stream));
  h->launches += 1;
  return SW_OK;
}

static size_t blob_size(sw_handle* h, int nf) {
  return sizeof(BlobHeader) + (size_t)2 * nf * h->g.ms * 2 * h->tsz;
}

extern "C" int sw_get_state(sw_handle* h, void* blob, size_t* size) {
  if (!h) return SW_EINVAL;
  h->err.clear();
  if (!size) return fail(h, SW_EINVAL, "size is NULL");
  const int nf = h->L.nf;
  const size_t need = blob_size(h, nf);
  if (!blob) {
    *size = need;
    return SW_OK;
  }
  if (*size < need) return fail(h, SW_EINVAL, "blob too small");
  BlobHeader hd;
  std::memset(&hd, 0, sizeof(hd));
  std::memcpy(hd.magic, "LAGMEAN1", 8);
  hd.version = 1;
  hd.N = h->p.N; hd.precision = h->p.precision; hd.model = h->p.model;
  hd.dt = h->p.dt; hd.f0 = h->p.f0; hd.c2 = h->p.c2; hd.nu8 = h->p.nu8; hd.lm_nu8 = h->p.lm_nu8;
  hd.adv_x = h->p.adv_x; hd.adv_y = h->p.adv_y;
  hd.stepper = h->p.stepper; hd.visc = h->p.visc;
  hd.lm_open = h->lm_open ? 1 : 0;
  hd.nf = nf;
  hd.lp = h->lp;
  hd.done = h->done;
  hd.steps_total = h->steps_total;
  std::memcpy(blob, &hd, sizeof(hd));
  if (const int rc = spec_rows(h, nf, true)) return rc;
  CK(h, cudaMemcpyAsync((char*)blob + sizeof(hd), h->mix, need - sizeof(hd), cudaMemcpyDeviceToHost, h->stream));
  CK(h, cudaStreamSynchronize(h->stream));
  *size = need;
  return SW_OK;
}

extern "C" int sw_set_state(sw_handle* h, const void* blob, size_t size) {
  if (!h) return SW_EINVAL;
  h->err.clear();
  if (!blob || size < sizeof(BlobHeader)) return fail(h, SW_EINVAL, "blob too small");
  BlobHeader hd;
  std::memcpy(&hd, blob, sizeof(hd));
  if (std::memcmp(hd.magic, "LAGMEAN1", 8) != 0 || hd.version != 1) return fail(h, SW_EINVAL, "not a state blob");
  if (hd.N != h->p.N || hd.precision != h->p.precision || hd.model != h->p.model || hd.dt != h->p.dt ||
      hd.f0 != h->p.f0 || hd.c2 != h->p.c2 || hd.nu8 != h->p.nu8 || hd.lm_nu8 != h->p.lm_nu8 ||
      hd.adv_x != h->p.adv_x || hd.adv_y != h->p.adv_y || hd.stepper != h->p.stepper || hd.visc != h->p.visc)
    return fail(h, SW_EINVAL, "blob parameters differ from the handle's");
  Layout L = hd.lm_open ? build_layout(h->p, hd.lp.strategy, hd.lp.fields, hd.lp.eulerian, hd.lp.scheme)
                        : build_layout(h->p, 0, 0, 0);
  if (L.nf != hd.nf || size < blob_size(h, hd.nf)) return fail(h, SW_EINVAL, "blob size mismatch");
  // (in halves of at most 64 KB where that lets the copies go with the commands)
  const size_t bytes = blob_size(h, hd.nf) - sizeof(hd), half = bytes / 2;
  const size_t first = bytes > (64 << 10) && half <= (64 << 10) ? half : bytes;
  const char* src = (const char*)blob + sizeof(hd);
  CK(h, cudaMemcpyAsync(h->mix, src, first, cudaMemcpyHostToDevice, h->stream));
  if (first < bytes)
    CK(h, cudaMemcpyAsync((char*)h->mix + first, src + first, bytes - first, cudaMemcpyHostToDevice, h->stream));
  if (const int rc = spec_rows(h, hd.nf, false, hd.done)) return rc;
  CK(h, cudaStreamSynchronize(h->stream));
  set_layout(h, L);
  h->lm_open = hd.lm_open != 0;
  h->lp = hd.lp;
  h->done = hd.done;
  h->steps_total = hd.steps_total;
  return SW_OK;
}

extern "C" int sw_spectrum(sw_handle* h, const double* field, int on_device, double* spectrum, int nshell) {
  if (!h) return SW_EINVAL;
  h->err.clear();
  if (!field || !spectrum) return fail(h, SW_EINVAL, "field and spectrum are required");
  const Geom& g = h->g;
  const int ns = (int)std::floor(std::sqrt(2.0) * g.K + 0.5) + 1;
  if (nshell < ns)
    return fail(h, SW_EINVAL, "nshell must be at least round(sqrt(2) K) + 1 = " + std::to_string(ns));
  cudaStream_t s = h->stream;
  // the field into the FP64 staging slot 0, forward 2D transform into the
  // spectral staging slot 0 (the path of an initial condition), shell sums
  // into staging slot 1
  CK(h, cudaMemcpyAsync(h->out64, field, (size_t)g.np * sizeof(double),
                        on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s));
  InArgs<double> ia;
  std::memset(&ia, 0, sizeof(ia));
  ia.phys = h->out64;
  ia.mix = h->mix64;
  ia.y = h->spec64;
  ia.tw = h->tw64;
  ia.g = g;
  ia.n = 1;
  CK(h, launch_in<double>(ia, s));
  double* acc = h->out64 + g.np;
  CK(h, cudaMemsetAsync(acc, 0, (size_t)ns * sizeof(double), s));
  CK(h, launch_spectrum_shells(h->spec64, g, acc, s));
  h->launches += 3;
  std::vector<double> tmp(ns);
  CK(h, cudaMemcpyAsync(tmp.data(), acc, (size_t)ns * sizeof(double), cudaMemcpyDeviceToHost, s));
  CK(h, cudaStreamSynchronize(s));
  for (int k = 0; k < nshell; ++k) spectrum[k] = k < ns ? tmp[k] : 0.0;
  return SW_OK;
}

extern "C" int sw_kernel_times(sw_handle* h, int64_t nsteps, double ms[SW_K_COUNT], int64_t launches[SW_K_COUNT],
                               double bytes[SW_K_COUNT]) {
  if (!h) return SW_EINVAL;
  h->err.clear();
  if (!ms || !launches || !bytes) return fail(h, SW_EINVAL, "output arrays are NULL");
  if (nsteps < 1) return fail(h, SW_EINVAL, "nsteps must be >= 1");
  if (h->lm_open && nsteps > h->lp.n_steps - h->done) return fail(h, SW_ERANGE, "more steps than remain in the interval");
  for (int k = 0; k < SW_K_COUNT; ++k) {
    ms[k] = 0.0;
    launches[k] = 0;
    bytes[k] = 0.0;
  }
  BatchExec* b = h->self;
  if (batch_stale(b)) {
    int rc = batch_build(b);
    if (rc) return fail(h, rc, b->err);
  }
  Prof pf;
  int nev = 0;
  cudaError_t e = cudaSuccess;
  for (; nev < 2 * Prof::MAXEV; ++nev)
    if ((e = cudaEventCreate(&pf.ev[nev])) != cudaSuccess) break;
  int rc = SW_OK;
  if (e != cudaSuccess) rc = fail_cuda(h, "cudaEventCreate", e);
  for (int64_t it = 0; rc == SW_OK && it < nsteps; ++it) {
    pf.n = 0;
    int64_t nl = 0;
    if (it == 0) {
      e = h->fp32 ? enqueue_batch_start<float>(b, h->stream, &pf, &nl) : enqueue_batch_start<double>(b, h->stream, &pf, &nl);
      if (e != cudaSuccess) {
        rc = fail_cuda(h, "sw_kernel_times start", e);
        break;
      }
    }
    const bool fin = it == nsteps - 1;
    e = h->fp32 ? enqueue_batch_step<float>(b, fin, h->stream, &pf, &nl)
                : enqueue_batch_step<double>(b, fin, h->stream, &pf, &nl);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) {
      rc = fail_cuda(h, "sw_kernel_times step", e);
      break;
    }
    h->launches += nl;
    h->steps_total += 1;
    if (h->lm_open) h->done += 1;
    for (int i = 0; i < pf.n; ++i) {
      float t = 0.f;
      if ((e = cudaEventElapsedTime(&t, pf.ev[2 * i], pf.ev[2 * i + 1])) != cudaSuccess) {
        rc = fail_cuda(h, "cudaEventElapsedTime", e);
        break;
      }
      ms[pf.cls[i]] += t;
      launches[pf.cls[i]] += 1;
      bytes[pf.cls[i]] += pf.bytes[i];
    }
  }
  for (int i = 0; i < nev; ++i) cudaEventDestroy(pf.ev[i]);
  return rc;
}

// ---------------------------------------------------------------------------
// Batches
struct sw_batch {
  BatchExec* ex = nullptr;
  std::string err;
  int tuned = -1;
};

static int bfail(sw_batch* b, int code, const std::string& msg) {
  b->err = msg;
  return code;
}

extern "C" int sw_batch_create(sw_handle* const* handles, int n, sw_batch** out) {
  g_create_error.clear();
  if (!out) return fail(nullptr, SW_EINVAL, "out is NULL");
  *out = nullptr;
  if (!handles || n < 1) return fail(nullptr, SW_EINVAL, "a batch needs at least one handle");
  for (int i = 0; i < n; ++i) {
    if (!handles[i]) return fail(nullptr, SW_EINVAL, "NULL handle in batch");
    for (int j = 0; j < i; ++j)
      if (handles[j] == handles[i]) return fail(nullptr, SW_EINVAL, "handle repeated in batch");
    if (handles[i]->fp32 != handles[0]->fp32) return fail(nullptr, SW_EINVAL, "batch members differ in precision");
    if (handles[i]->stream != handles[0]->stream) return fail(nullptr, SW_EINVAL, "batch members differ in stream");
  }
  sw_batch* b = new (std::nothrow) sw_batch();
  BatchExec* ex = b ? new (std::nothrow) BatchExec() : nullptr;
  if (!ex) {
    delete b;
    return fail(nullptr, SW_ENOMEM, "host allocation failed");
  }
  b->ex = ex;
  ex->members.assign(handles, handles + n);
  ex->fp32 = handles[0]->fp32;
  ex->stream = handles[0]->stream;
  int rc = batch_build(ex);
  if (rc != SW_OK) {
    std::string m = ex->err;
    batch_free(ex);
    delete b;
    return fail(nullptr, rc, m);
  }
  *out = b;
  return SW_OK;
}

extern "C" int sw_batch_step(sw_batch* b, int64_t nsteps) {
  if (!b) return SW_EINVAL;
  b->err.clear();
  if (nsteps < 0) return bfail(b, SW_EINVAL, "nsteps < 0");
  for (sw_handle* h : b->ex->members)
    if (h->lm_open && nsteps > h->lp.n_steps - h->done)
      return bfail(b, SW_ERANGE, "more steps than remain in a member's interval");
  if (nsteps == 0) return SW_OK;
  int rc = batch_replay(b->ex, nsteps);
  if (rc) return bfail(b, rc, b->ex->err);
  for (sw_handle* h : b->ex->members) {
    h->steps_total += nsteps;
    if (h->lm_open) h->done += nsteps;
  }
  return SW_OK;
}

// Save / restore the evolving state of the members around tuning trials.
struct Saved {
  void* buf = nullptr;
  size_t fb = 0;
  long long ctr = 0;
};

extern "C" int sw_batch_tune(sw_batch* b, int trial_steps, int* choice) {
  if (!b) return SW_EINVAL;
  b->err.clear();
  if (trial_steps < 1) return bfail(b, SW_EINVAL, "trial_steps must be >= 1");
  BatchExec* ex = b->ex;
  int maxN = 0;
  for (sw_handle* h : ex->members) maxN = h->g.N > maxN ? h->g.N : maxN;
  const int pts[4] = {256, 512, 1024, 2048};
  const int ppbs[4] = {1, 2, 3, MAXP};
  std::vector<Saved> saved(ex->members.size());
  cudaError_t e = cudaSuccess;
  int rc = SW_OK;
  for (size_t i = 0; i < ex->members.size() && rc == SW_OK; ++i) {
    sw_handle* h = ex->members[i];
    saved[i].fb = (size_t)MAXF * h->g.ms * 2 * h->tsz;
    if ((e = cudaMalloc(&saved[i].buf, 2 * saved[i].fb)) != cudaSuccess) {
      cudaGetLastError();
      saved[i].buf = nullptr;
      rc = bfail(b, SW_ENOMEM, std::string("cudaMalloc (tuning copy): ") + cudaGetErrorString(e));
      break;
    }
    if ((e = cudaMemcpyAsync(saved[i].buf, h->y, saved[i].fb, cudaMemcpyDeviceToDevice, ex->stream)) != cudaSuccess ||
        (e = cudaMemcpyAsync((char*)saved[i].buf + saved[i].fb, h->comp, saved[i].fb, cudaMemcpyDeviceToDevice,
                             ex->stream)) != cudaSuccess ||
        (e = cudaMemcpyAsync(&saved[i].ctr, h->ctr, sizeof(long long), cudaMemcpyDeviceToHost, ex->stream)) != cudaSuccess)
      rc = bfail(b, SW_ECUDA, std::string("tuning save: ") + cudaGetErrorString(e));
  }
  if (rc == SW_OK && (e = cudaStreamSynchronize(ex->stream)) != cudaSuccess)
    rc = bfail(b, SW_ECUDA, std::string("tuning save: ") + cudaGetErrorString(e));
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (rc == SW_OK && ((e = cudaEventCreate(&e0)) != cudaSuccess || (e = cudaEventCreate(&e1)) != cudaSuccess))
    rc = bfail(b, SW_ECUDA, std::string("cudaEventCreate: ") + cudaGetErrorString(e));
  int best = -1;
  float best_ms = 0.f;
  for (int ci = 0; rc == SW_OK && ci < 16; ++ci) {
    const int P = pts[ci / 4], ppb = ppbs[ci % 4];
    if (P < maxN) continue;  // every member needs rows x N = P (equal block shapes)
    for (sw_handle* h : ex->members) {
      h->points = P;
      h->ppb = ppb;
      ++h->version;
    }
    rc = batch_ready(ex);
    // untimed replay of the same steps first: a new graph's first launch
    // carries its upload, which would bias the trials
    if (rc == SW_OK) rc = batch_replay(ex, trial_steps);
    if (rc) {
      rc = bfail(b, rc, ex->err);
      break;
    }
    if ((e = cudaEventRecord(e0, ex->stream)) != cudaSuccess) break;
    rc = batch_replay(ex, trial_steps);
    if (rc) {
      rc = bfail(b, rc, ex->err);
      break;
    }
    if ((e = cudaEventRecord(e1, ex->stream)) != cudaSuccess || (e = cudaEventSynchronize(e1)) != cudaSuccess) break;
    float t = 0.f;
    if ((e = cudaEventElapsedTime(&t, e0, e1)) != cudaSuccess) break;
    if (best < 0 || t < best_ms) {
      best = ci;
      best_ms = t;
    }
  }
  if (rc == SW_OK && e != cudaSuccess) rc = bfail(b, SW_ECUDA, std::string("tuning trial: ") + cudaGetErrorString(e));
  if (best < 0) {  // no trial ran: a shape every member fits (512 points or one row pair, all products)
    int pi = 1;
    while (pi < 3 && pts[pi] < maxN) ++pi;
    best = 4 * pi + 3;
  }
  for (sw_handle* h : ex->members) {
    h->points = pts[best / 4];
    h->ppb = ppbs[best % 4];
    ++h->version;
  }
  // restore the saved states
  for (size_t i = 0; i < ex->members.size(); ++i) {
    sw_handle* h = ex->members[i];
    if (!saved[i].buf) continue;
    if (rc == SW_OK) {
      if ((e = cudaMemcpyAsync(h->y, saved[i].buf, saved[i].fb, cudaMemcpyDeviceToDevice, ex->stream)) != cudaSuccess ||
          (e = cudaMemcpyAsync(h->comp, (char*)saved[i].buf + saved[i].fb, saved[i].fb, cudaMemcpyDeviceToDevice,
                               ex->stream)) != cudaSuccess ||
          (e = cudaMemcpyAsync(h->ctr, &saved[i].ctr, sizeof(long long), cudaMemcpyHostToDevice, ex->stream)) != cudaSuccess)
        rc = bfail(b, SW_ECUDA, std::string("tuning restore: ") + cudaGetErrorString(e));
    }
  }
  cudaError_t es = cudaStreamSynchronize(ex->stream);
  if (rc == SW_OK && es != cudaSuccess) rc = bfail(b, SW_ECUDA, std::string("tuning restore: ") + cudaGetErrorString(es));
  for (auto& sv : saved)
    if (sv.buf) cudaFree(sv.buf);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  b->tuned = best;
  if (choice) *choice = best;
  return rc;
}

extern "C" int sw_batch_set_shape(sw_batch* b, int choice) {
  if (!b) return SW_EINVAL;
  b->err.clear();
  static const int pts[4] = {256, 512, 1024, 2048};
  static const int ppbs[4] = {1, 2, 3, MAXP};
  if (choice < 0 || choice >= 16) return bfail(b, SW_EINVAL, "choice must be in 0..15");
  BatchExec* ex = b->ex;
  for (sw_handle* h : ex->members)
    if (pts[choice / 4] < h->g.N) return bfail(b, SW_EINVAL, "points per block below a member's N");
  for (sw_handle* h : ex->members) {
    h->points = pts[choice / 4];
    h->ppb = ppbs[choice % 4];
    ++h->version;
  }
  b->tuned = choice;
  return SW_OK;
}

extern "C" int sw_batch_launch_count(sw_batch* b, int64_t* count) {
  if (!b || !count) return SW_EINVAL;
  *count = b->ex->launches;
  return SW_OK;
}

extern "C" const char* sw_batch_last_error(sw_batch* b) { return b ? b->err.c_str() : ""; }

extern "C" void sw_batch_destroy(sw_batch* b) {
  if (!b) return;
  if (b->ex) cudaStreamSynchronize(b->ex->stream);
  batch_free(b->ex);
  delete b;
}

extern "C" int sw_launch_count(sw_handle* h, int64_t* count) {
  if (!h || !count) return SW_EINVAL;
  *count = h->launches;
  return SW_OK;
}

extern "C" int sw_time(sw_handle* h, double* t) {
  if (!h || !t) return SW_EINVAL;
  *t = (double)h->steps_total * h->p.dt;
  return SW_OK;
}

extern "C" int sw_sync(sw_handle* h) {
  if (!h) return SW_EINVAL;
  CK(h, cudaStreamSynchronize(h->stream));
  return SW_OK;
}

extern "C" const char* sw_last_error(sw_handle* h) { return h ? h->err.c_str() : g_create_error.c_str(); }

extern "C" const char* sw_version(void) { return "lagmean-gb300 0.1"; }
