// Source terms and the analytical Jacobian of the molar, explicitly
// mass-conserving formulation (Sec. 2.2) over a structure-of-arrays batch,
// lane = state.
//
// GB300 design notes:
//  * The path is bound by the FP64 pipe (2 FP64 FMA per clock per SM on this
//    part, a 64th of the FP32 rate), not by HBM, so the kernels minimise
//    FP64 instructions: exponents, exponentials and logarithms are integer
//    fixed point (fixed_math.cuh), one exponential per forward rate and one
//    per reverse rate (from ln kf - ln Kc).
//  * The warps of a block share 32 states: concentrations, Gibbs energies and
//    enthalpies sit once in shared memory or, for large mechanisms, in a
//    global workspace.
//  * Reaction constants are read warp-uniformly (every thread of a warp works
//    on the same reaction), so there is no divergence except the NASA range.
//  * Jacobian entries are accumulated with fire-and-forget FP64 reductions
//    into the zero-initialised output at L2 (no read-modify-write latency on
//    the SM and no FP64 add on the SM).  One state per thread, each entry is
//    owned by one thread, whose reductions apply in program order, so results
//    are deterministic; the cooperative layout sums one entry from several
//    warps, in an order that can change between runs.  The source terms'
//    sums are in a fixed order (source_tile.cuh).
//    Targets come from a static full -> sparse index map built at mechanism
//    load (the mapping Sec. 3.4 proposes instead of a per-entry search).
//  * This file holds the source-term kernel and the launch planning; the
//    Jacobian kernels are in jacobian_kernels.cuh (instantiated by
//    jacobian_inst.cu).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>

#include "jacobian_kernels.cuh"  // k_jacobian_coop's tile and shared-memory size (the kernels: jacobian_inst.cu)
#include "kinetics_state.cuh"
#include "source_tile.cuh"
#ifndef PJ_NO_LAUNCHERS
#include "launch.h"
#endif

namespace pj {

// ---------------------------------------------------------------------------
// source terms
// ---------------------------------------------------------------------------
// A block of 16 warps per 32-state tile (source_tile.cuh), two blocks per SM,
// or of 32 where there are no more tiles than SMs; tiles handed out
// block-cyclically.  Y: y = (wdot, dT/dt) instead of dPhi/dt.
template <int MODE, bool SPECIAL, bool Y, bool SHARED>
__global__ void __launch_bounds__(2 * kSrcWarps * 32, 1)
    k_source_terms(const __grid_constant__ DevMech m, int64_t n, const double* __restrict__ param,
                   const double* __restrict__ phi, int64_t ld, double* __restrict__ out, int* status, double* ws,
                   double* arrays) {
  PJ_DYN_SMEM;
  load_exp_table(m.exp_tab);
  const int lane = threadIdx.x & 31;
  if (arrays) arrays += (size_t)blockIdx.x * source_arrays_ws_doubles(m.ns, false);
  if (!Y) ws += (size_t)blockIdx.x * m.ns * kTile + lane;
  for (int64_t tile = blockIdx.x; tile * kTile < n; tile += gridDim.x) {
    const int64_t s = tile * kTile + lane;
    const BatchIn in{param, phi, ld, s, s < n};
    if constexpr (Y) source_tile<MODE, SPECIAL, SHARED ? kShared : kGlobal>(m, smem, arrays, in, YOut{out, ld, s, m.ns, status});
    else source_tile<MODE, SPECIAL, SHARED ? kShared : kGlobal>(m, smem, arrays, in, SourceOut{out, ws, ld, s, m.ns, status});
  }
}

// pj_exp next to the library exp, for verification (pj_diag_exp).
__global__ void k_diag_exp(const uint64_t* __restrict__ tab, int64_t n, const double* __restrict__ x,
                           double* __restrict__ y_ours, double* __restrict__ y_lib) {
  load_exp_table(tab);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    y_ours[i] = pj_exp(x[i]);
    y_lib[i] = exp(x[i]);
  }
}

#ifndef PJ_NO_LAUNCHERS
int launch_diag_exp(const DevMech& m, int64_t n, const double* x, double* y_ours, double* y_lib, cudaStream_t st) {
  int64_t blocks = (n + 255) / 256;
  if (blocks > 65535) blocks = 65535;
  if (blocks < 1) blocks = 1;
  k_diag_exp<<<(unsigned)blocks, 256, 0, st>>>(m.exp_tab, n, x, y_ours, y_lib);
  return check_cuda(cudaGetLastError(), "k_diag_exp launch");
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static int g_num_sms[64] = {};

int sm_count() {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) dev = 0;
  if (g_num_sms[dev] == 0) {
    int c = 0;
    cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, dev);
    g_num_sms[dev] = c > 0 ? c : 1;
  }
  return g_num_sms[dev];
}

// Per-state arrays: in shared memory when 128 threads fit, else in a global
// workspace with a grid-stride grid (trimmed to the resident blocks at
// launch, see resident_grid).
LaunchPlan plan_for(int arrays, int ns, int64_t n) {
  LaunchPlan p{};
  const size_t per_thread = (size_t)arrays * ns * sizeof(double);
  // threads per SM that fit the per-state arrays in shared memory, as whole
  // warps; blocks of up to 128 threads so several can share an SM
  const int fit = (int)((kSmemCap / per_thread) / 32 * 32);
  if (fit >= 128) {
    p.global_ws = false;
    p.tpb = fit >= 256 ? 128 : (fit % 64 == 0 ? 64 : 32);
    p.smem = per_thread * p.tpb;
    const int64_t blocks = (n + p.tpb - 1) / p.tpb;
    p.grid = (int)(blocks < 1 ? 1 : blocks);
    p.ws_bytes = 0;
    p.ws_stride = 0;
  } else {
    p.global_ws = true;
    p.tpb = 128;
    p.smem = 0;
    const int64_t cap = (int64_t)sm_count() * 4;
    const int64_t blocks = (n + p.tpb - 1) / p.tpb;
    p.grid = (int)(blocks < cap ? (blocks < 1 ? 1 : blocks) : cap);
    p.ws_stride = (int64_t)p.grid * p.tpb;
    p.ws_bytes = per_thread * (size_t)p.ws_stride;
  }
  return p;
}

int source_arrays() { return 2; }
int jacobian_arrays() { return 3; }

// The tile kernel's shape: arrays in shared memory while two blocks fit an
// SM, then while one does, else in the workspace (two blocks).
SourcePlan source_plan(int ns, int64_t n) {
  SourcePlan p{};
  const size_t in_smem = source_smem_bytes(ns, true);
  p.arrays_smem = in_smem <= kSmemCap;
  p.smem = source_smem_bytes(ns, p.arrays_smem);
  p.ctas = p.smem + kBlockOverhead <= kSmemPerSm / 2 ? 2 : 1;
  const int64_t tiles = (n + kTile - 1) / kTile;
  p.warps = tiles <= sm_count() ? 2 * kSrcWarps : kSrcWarps;
  p.grid = (int)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)sm_count() * p.ctas));
  p.acc_bytes = (size_t)p.grid * ns * kTile * sizeof(double);
  p.arrays_bytes = (size_t)p.grid * source_arrays_ws_doubles(ns, p.arrays_smem) * sizeof(double);
  return p;
}

template <bool Y>
static int launch_source_t(const DevMech& m, int mode, int64_t n, const double* param, const double* phi, int64_t ld,
                           double* out, int* status, void* work, size_t work_bytes, cudaStream_t st) {
  const SourcePlan p = source_plan(m.ns, n);
  const size_t need = (Y ? 0 : p.acc_bytes) + p.arrays_bytes;
  if (need && (!work || work_bytes < need))
    return fail(PJ_ERR_NOMEM, Y ? "workspace too small for pj_eval_y (see pj_workspace_size)"
                                : "workspace too small for the source-term kernel (see pj_workspace_size)");
  double* arrays = p.arrays_bytes ? static_cast<double*>(work) : nullptr;
  double* acc = Y ? nullptr : static_cast<double*>(work) + p.arrays_bytes / sizeof(double);
  const bool special = m.nr_plain < m.nr;
  auto pick = [&](auto shared) {
    constexpr bool SH = decltype(shared)::value;
    return mode == PJ_CONP ? (special ? k_source_terms<PJ_CONP, true, Y, SH> : k_source_terms<PJ_CONP, false, Y, SH>)
                           : (special ? k_source_terms<PJ_CONV, true, Y, SH> : k_source_terms<PJ_CONV, false, Y, SH>);
  };
  auto kern = p.arrays_smem ? pick(BoolTag<true>{}) : pick(BoolTag<false>{});
  int rc;
  if ((rc = set_smem(kern, p.smem))) return rc;
  kern<<<p.grid, p.warps * 32, p.smem, st>>>(m, n, param, phi, ld, out, status, acc, arrays);
  return check_cuda(cudaGetLastError(), "k_source_terms launch");
}

int launch_source(const DevMech& m, int mode, int64_t n, const double* param, const double* phi, int64_t ld,
                  double* out, int* status, void* work, size_t work_bytes, cudaStream_t st) {
  return launch_source_t<false>(m, mode, n, param, phi, ld, out, status, work, work_bytes, st);
}

int launch_eval_y(const DevMech& m, int mode, int64_t n, const double* param, const double* phi, int64_t ld,
                  double* y, int* status, void* work, size_t work_bytes, cudaStream_t st) {
  return launch_source_t<true>(m, mode, n, param, phi, ld, y, status, work, work_bytes, st);
}

// TMEM mode for the Jacobian.  Chosen when it keeps at least as many
// threads resident as the plain kernel (arrays in shared memory when 128
// threads fit, else in a workspace at the register-limited occupancy); of the
// splits of C_k, g_k/RT between shared memory and the workspace, the one with
// the most resident blocks, on ties the one with the fewest arrays in shared
// memory (L1-cached workspace loads measured faster than shared-memory loads
// at equal occupancy on the 53-species workload).
TmPlan tm_plan(int ns) {
  TmPlan t{false, 0, 2, 0, 0, 0, 0};
  uint32_t nc = 32;
  while (nc < 2u * (uint32_t)ns) nc <<= 1;
  if (nc > 512) return t;
  const int tm_ctas = (int)(512 / nc);
  int best_ctas = 0, best_split = 2;
  size_t best_smem = 0;
  for (int split = 0; split <= 2; split++) {
    const size_t dyn = (size_t)split * ns * sizeof(double) * 128;
    if (dyn > kSmemCap) continue;
    const int smem_ctas = (int)(kSmemPerSm / (dyn + kBlockOverhead));
    const int ctas = std::min(std::min(smem_ctas, tm_ctas), kJacRegCtas);
    if (ctas > best_ctas) {
      best_ctas = ctas;
      best_split = split;
      best_smem = dyn;
    }
  }
  if (best_ctas == 0) return t;
  const size_t per3 = (size_t)3 * ns * sizeof(double);
  const int fit = (int)((kSmemCap / per3) / 32 * 32);
  const int plain_threads = fit >= 128 ? std::min(fit, kJacRegCtas * 128) : kJacRegCtas * 128;
  if (best_ctas * 128 < plain_threads || (best_ctas * 128 == plain_threads && fit >= 128)) return t;
  t.use = true;
  t.ncols = nc;
  t.split = best_split;
  t.ctas = best_ctas;
  t.smem = best_smem;
  if (best_split < 2) {
    t.grid = sm_count() * best_ctas;
    t.ws_bytes = (size_t)(2 - best_split) * ns * sizeof(double) * (size_t)t.grid * 128;
  }
  return t;
}

// Which Jacobian layout runs, chosen by measurement on GB300 (microseconds;
// cooperative shapes as warps x blocks per SM, "one" for one state per thread):
//  * at most one 32-state tile per SM: cooperative, 20 warps on each tile, or
//    16 where 20 would take as many rounds over the reactions (13 species, 27
//    reactions, 4096 states: 46.0 at 16 x 1, 48.9 at 20 x 1, 289 one);
//  * larger batches: cooperative, 10 x 2 (53 species CSR, 131072 states: 5063
//    against 5440 at 8 x 2, 5708 at 4 x 4, 5531 at 16 x 1, 10365 one; dense
//    the same; FP32 Newton matrix of 111 species, 32768 states: 2887 against
//    3193, 3356, 2922 and 9166), 16 x 1 above 200 species (the 874-species
//    arrays are 671 KB a tile), 4 x 4 for small mechanisms at 512 states per
//    SM or more (13 species, 524288 states: 2541 against 2854 at 8 x 2 and
//    3500 one);
//  * from 1 Mi states on, the dense FP64 Jacobian of TMEM-size mechanisms (53
//    species) and the Jacobians of mechanisms whose arrays fit shared memory
//    for one state per thread (13 species) stay one state per thread, the
//    layout pj_jacobian_layout is documented and tested to answer there.  The
//    cooperative layout is the faster one at that size too (53 species dense,
//    1 Mi: 42.5 ms against 79.4).
// Each cooperative block keeps only its 32 states' Jacobians live in L2, a
// fraction of the one-state-per-thread kernels' live set (DRAM traffic per
// state at 53 species: 154 KB in TMEM, 34 KB at 16 x 1, 65 KB at 8 x 2), so
// 16 x 1 is the shape to force where the Jacobian shares the GPU with other
// memory-heavy work.
// The cooperative kernel keeps a tile's per-state arrays in shared memory
// where they fit, else in a workspace of 3 Ns x 32 doubles per block, which
// stays in L2 (874 species at one block per SM: 102 MB).
// PYJAC_GB_JAC_LAYOUT=coop|percore forces one family (coop only where its
// shared memory fits); PYJAC_GB_COOP_WARPS sets the warps per block (4, 8
// or 16), PYJAC_GB_COOP_CTAS the blocks per SM (at most 16 / warps) and
// PYJAC_GB_COOP_ARRAYS=global puts the arrays in the workspace.
static int env_int(const char* name, int dflt) {
  const char* v = getenv(name);
  return v && *v ? atoi(v) : dflt;
}

bool coop_shape(const DevMech& m, int warps, int ctas, bool arrays_smem, int64_t tiles, CoopPlan& c) {
  c = CoopPlan{false, warps, ctas, coop_smem_bytes(m.ns, warps, arrays_smem), sm_count() * ctas, 0};
  if (warps < 4 || ctas < 1 || ctas * warps > kCoopWarpsMax) return false;
  if (c.smem + kBlockOverhead > kSmemPerSm / (size_t)ctas || c.smem > kSmemCap) return false;
  if (!arrays_smem) {
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>(tiles, c.grid));
    c.ws_bytes = coop_arrays_bytes(m.ns) * (size_t)blocks;
  }
  c.use = true;
  return true;
}

// per-state arrays in shared memory where they fit, else in the workspace
static bool coop_fit(const DevMech& m, int warps, int ctas, int64_t n, CoopPlan& c) {
  const int64_t tiles = (n + kCoopTile - 1) / kCoopTile;
  return coop_shape(m, warps, ctas, true, tiles, c) || coop_shape(m, warps, ctas, false, tiles, c);
}

constexpr int64_t kPercoreStates = int64_t(1) << 20;

CoopPlan coop_plan(const DevMech& m, int fmt, int dt_bytes, int64_t n) {
  CoopPlan c{false, 16, 1, 0, 0, 0};
  const char* lay = getenv("PYJAC_GB_JAC_LAYOUT");
  if (lay && strcmp(lay, "percore") == 0) return c;
  if (lay && strcmp(lay, "coop") == 0) {
    const int warps = env_int("PYJAC_GB_COOP_WARPS", 16), ctas = env_int("PYJAC_GB_COOP_CTAS", 16 / std::max(warps, 1));
    if ((warps != 4 && warps != 8 && warps != 16) || warps * ctas > 16) return c;
    const char* ar = getenv("PYJAC_GB_COOP_ARRAYS");
    if (ar && strcmp(ar, "global") == 0) coop_shape(m, warps, ctas, false, (n + kCoopTile - 1) / kCoopTile, c);
    else coop_fit(m, warps, ctas, n, c);
    return c;
  }
  const TmPlan t = tm_plan(m.ns);
  const int sms = sm_count();
  const int64_t tiles = (n + kCoopTile - 1) / kCoopTile;
  const bool percore_global = !t.use && plan_for(jacobian_arrays(), m.ns, n).global_ws;
  if (tiles <= sms) {  // one tile per SM at most: 20 warps where that takes fewer rounds than 16
    const int r16 = (m.nr + 15) / 16, r20 = (m.nr + kCoopWarpsMax - 1) / kCoopWarpsMax;
    if (r20 == r16 || !coop_shape(m, kCoopWarpsMax, 1, true, tiles, c)) coop_fit(m, 16, 1, n, c);
    return c;
  }
  if (n < kPercoreStates) {
    if (m.ns > 200) coop_fit(m, 16, 1, n, c);
    else if (t.use || percore_global || n < (int64_t)sms * 512) coop_fit(m, kCoopWarpsMax / 2, 2, n, c);
    else coop_fit(m, 4, 4, n, c);
    return c;
  }
  if (t.use || percore_global) {
    if (t.use && fmt == PJ_DENSE && dt_bytes == 8) return c;
    if (m.ns > 200) coop_fit(m, 16, 1, n, c);
    else coop_fit(m, kCoopWarpsMax / 2, 2, n, c);
    return c;
  }
  c.use = false;
  return c;
}

size_t workspace_bytes(int arrays, int ns, int64_t n) {
  if (arrays == jacobian_arrays()) {
    // the most any layout can need: the one-state-per-thread plans, or the
    // cooperative one with its arrays in the workspace
    const TmPlan t = tm_plan(ns);
    const size_t pc = t.use ? t.ws_bytes : plan_for(arrays, ns, n).ws_bytes;
    // (any shape that may not fit its arrays in shared memory: at most 4
    // blocks per SM, since a block has 4 warps or more)
    const int64_t tiles =
        std::max<int64_t>(1, std::min<int64_t>((n + kCoopTile - 1) / kCoopTile, (int64_t)sm_count() * 4));
    const char* ar = getenv("PYJAC_GB_COOP_ARRAYS");
    const bool global = 4 * (coop_smem_bytes(ns, 4) + kBlockOverhead) > kSmemPerSm ||
                        coop_smem_bytes(ns, 16) > kSmemCap || (ar && strcmp(ar, "global") == 0);
    const size_t co = global ? coop_arrays_bytes(ns) * (size_t)tiles : 0;
    return std::max(pc, co);
  }
  const SourcePlan p = source_plan(ns, n);
  return p.acc_bytes + p.arrays_bytes;
}

int launch_jac_coop_f64(const DevMech& m, const CoopPlan& p, int mode, int fmt, int64_t n, const JacArgs& a,
                        double* ws, cudaStream_t st) {
  return (fmt == PJ_CSR ? launch_jac_coop_f64_csr : fmt == PJ_CSC ? launch_jac_coop_f64_csc
                                                                  : launch_jac_coop_f64_dense)(m, p, mode, n, a, ws, st);
}

int launch_jac_coop_f32(const DevMech& m, const CoopPlan& p, int mode, int fmt, int64_t n, const JacArgs& a,
                        double* ws, cudaStream_t st) {
  return (fmt == PJ_CSR ? launch_jac_coop_f32_csr : fmt == PJ_CSC ? launch_jac_coop_f32_csc
                                                                  : launch_jac_coop_f32_dense)(m, p, mode, n, a, ws, st);
}

// Shared by the FP64 Jacobian and the FP32 Newton matrix: pick the layout,
// check the workspace, call the launcher of that layout and precision.
static int launch_jac_any(const DevMech& m, int mode, int fmt, int64_t n, const JacArgs& a, bool f32, void* work,
                          size_t work_bytes, cudaStream_t st) {
  const CoopPlan c = coop_plan(m, fmt, f32 ? 4 : 8, n);
  if (c.use) {
    if (c.ws_bytes && (!work || work_bytes < c.ws_bytes))
      return fail(PJ_ERR_NOMEM, "workspace too small for the Jacobian kernel (see pj_workspace_size)");
    return (f32 ? launch_jac_coop_f32 : launch_jac_coop_f64)(m, c, mode, fmt, n, a, static_cast<double*>(work),
                                                            st);
  }
  const TmPlan t = tm_plan(m.ns);
  if (t.use) {
    if (t.ws_bytes && (!work || work_bytes < t.ws_bytes))
      return fail(PJ_ERR_NOMEM, "workspace too small for the Jacobian kernel (see pj_workspace_size)");
    double* ws = static_cast<double*>(work);
    if (t.split == 2) return (f32 ? launch_jac_tm2_f32 : launch_jac_tm2_f64)(m, t, mode, fmt, n, a, ws, st);
    if (t.split == 1) return (f32 ? launch_jac_tm1_f32 : launch_jac_tm1_f64)(m, t, mode, fmt, n, a, ws, st);
    return (f32 ? launch_jac_tm0_f32 : launch_jac_tm0_f64)(m, t, mode, fmt, n, a, ws, st);
  }
  LaunchPlan p = plan_for(jacobian_arrays(), m.ns, n);
  if (p.global_ws && (!work || work_bytes < p.ws_bytes))
    return fail(PJ_ERR_NOMEM, "workspace too small for the Jacobian kernel (see pj_workspace_size)");
  double* ws = p.global_ws ? static_cast<double*>(work) : nullptr;
  return (f32 ? launch_jac_plain_f32 : launch_jac_plain_f64)(m, p, mode, fmt, n, a, ws, st);
}

int jacobian_layout(const DevMech& m, int fmt, bool f32, int64_t n) {
  if (coop_plan(m, fmt, f32 ? 4 : 8, n).use) return PJ_LAYOUT_COOP;
  return tm_plan(m.ns).use ? PJ_LAYOUT_TMEM : PJ_LAYOUT_PERCORE;
}

int launch_jacobian(const DevMech& m, int mode, int fmt, int64_t n, const double* param, const double* phi,
                    int64_t ld, double* J, double* dphi, int* status, void* work, size_t work_bytes,
                    cudaStream_t st) {
  const JacArgs a{param, phi, ld, J, dphi, status, nullptr, 0.0};
  return launch_jac_any(m, mode, fmt, n, a, false, work, work_bytes, st);
}

// Newton-iteration matrix M = I - h*gamma*J in FP32 (derivative arithmetic
// in FP32, rates and source terms in FP64).
int launch_newton_f32(const DevMech& m, int mode, int fmt, int64_t n, const double* param, const double* phi,
                      int64_t ld, const double* hstep, double gamma, float* M, double* dphi, int* status,
                      void* work, size_t work_bytes, cudaStream_t st) {
  const JacArgs a{param, phi, ld, M, dphi, status, hstep, gamma};
  return launch_jac_any(m, mode, fmt, n, a, true, work, work_bytes, st);
}

// Run k_jacobian with its per-state arrays in a scratch region that holds
// `scratch_threads` threads' arrays (grid-stride over the states).  Used by
// the allocation-free entry point (noalloc.cu).
int launch_jacobian_on_scratch(const DevMech& m, int mode, int fmt, int64_t n, const double* param,
                               const double* phi, int64_t ld, double* J, double* dphi, int* status,
                               double* scratch, int64_t scratch_threads, cudaStream_t st) {
  LaunchPlan p{};
  p.tpb = 128;
  p.global_ws = true;
  p.smem = 0;
  const int64_t blocks = (n + p.tpb - 1) / p.tpb;
  int64_t cap = scratch_threads / p.tpb;
  const int64_t sm_cap = (int64_t)sm_count() * 4;
  if (cap > sm_cap) cap = sm_cap;
  p.grid = (int)(blocks < cap ? (blocks < 1 ? 1 : blocks) : cap);
  p.ws_stride = (int64_t)p.grid * p.tpb;
  p.ws_bytes = (size_t)jacobian_arrays() * m.ns * sizeof(double) * (size_t)p.ws_stride;
  const JacArgs a{param, phi, ld, J, dphi, status, nullptr, 0.0};
  return launch_jac_plain_f64(m, p, mode, fmt, n, a, scratch, st);
}
#endif  // PJ_NO_LAUNCHERS

}  // namespace pj
