// First-order forward finite-difference Jacobian: the comparator against
// which Sec. 3.5.2 measures the analytical Jacobian's speedup: the source
// terms at Phi and at Phi + h_j e_j for every column j,
// with delta_j = 2^-26 max(|Phi_j|, 2^-26 n_tot), n_tot = P V / (R T), and the
// realised step h_j = (Phi_j + delta_j) - Phi_j (the paper gives no step
// rule; 2^-26 is about the square root of the unit roundoff, and a power of
// two keeps the scaling exact).  Column j is (f(Phi + h_j e_j) - f(Phi)) / h_j,
// stored in the handle's pattern (sparse) or in full (dense).  Every
// evaluation is the source-term kernel's (source_tile, bit for bit), so the
// cost is N + 1 source-term evaluations per state.
#include <cuda_runtime.h>

#include <algorithm>

#include "kinetics_state.cuh"
#include "launch.h"
#include "source_tile.cuh"

namespace pj {

constexpr double kFdScale = 0x1p-26;

// The batch's states with variable j moved by its step (j < 0: as they are).
template <int MODE>
struct FdIn {
  BatchIn in;
  int j;
  double lo;  // kFdScale n_tot
  __device__ __forceinline__ bool act() const { return in.active; }
  __device__ __forceinline__ double moved(double x) const { return x + kFdScale * fmax(fabs(x), lo); }
  __device__ __forceinline__ double T() const { return j == 0 ? moved(in.T()) : in.T(); }
  __device__ __forceinline__ double S() const { return j == 1 ? moved(in.S()) : in.S(); }
  __device__ __forceinline__ double par() const { return in.par(); }
  __device__ __forceinline__ double n(int k) const { return j == k + 2 ? moved(in.n(k)) : in.n(k); }
};

// Column j of the Jacobian from the moved state's source terms; f0: the
// source terms of the state itself.
template <int FMT>
struct FdOut {
  const DevMech& m;
  double* __restrict__ J;
  double* f0;
  double* __restrict__ ws;
  int64_t ld, s;
  int j;
  double h;
  __device__ __forceinline__ double* acc(int k) const { return ws + k * kTile; }
  __device__ __forceinline__ void entry(int i, double f1) const {
    const int64_t e = jpos<FMT>(m, i, j);
    if (e >= 0) J[e * ld + s] = (f1 - __ldcg(f0 + (int64_t)i * ld + s)) / h;
  }
  __device__ __forceinline__ void species(int k, double V, double wk) const {
    if (k < m.ns - 1) entry(k + 2, __dmul_rn(V, wk));  // rounded, as the source terms are stored
  }
  __device__ __forceinline__ void head(double Tdot, double Sdot) const {
    entry(0, Tdot);
    entry(1, Sdot);
  }
  __device__ __forceinline__ void invalid() const {
    for (int i = 0; i < m.N; i++) entry(i, __longlong_as_double(0x7ff8000000000000ULL));
  }
};

template <int MODE, int FMT, bool SPECIAL>
__global__ void __launch_bounds__(kSrcWarps * 32, 2)
    k_fd_jacobian(const __grid_constant__ DevMech m, int64_t n, const double* __restrict__ param,
                  const double* __restrict__ phi, int64_t ld, double* __restrict__ J, double* dphi, int* status,
                  double* ws, double* arrays) {
  PJ_DYN_SMEM;
  load_exp_table(m.exp_tab);
  const int lane = threadIdx.x & 31;
  if (arrays) arrays += (size_t)blockIdx.x * source_arrays_ws_doubles(m.ns, false);
  ws += (size_t)blockIdx.x * m.ns * kTile + lane;
  for (int64_t tile = blockIdx.x; tile * kTile < n; tile += gridDim.x) {
    const int64_t s = tile * kTile + lane;
    const BatchIn in{param, phi, ld, s, s < n};
    source_tile<MODE, SPECIAL, kEither>(m, smem, arrays, in, SourceOut{dphi, ws, ld, s, m.ns, status});
    __syncthreads();  // the source terms of every row before any warp reads them
    double lo = 0.0;
    if (in.active) {
      const double T = in.T(), S = in.S(), par = in.par();
      const double V = MODE == PJ_CONP ? S : par, P = MODE == PJ_CONP ? par : S;
      lo = kFdScale * ((P * V) / (RU * T));
    }
    for (int j = 0; j < m.N; j++) {
      double h = 1.0;
      if (in.active) {
        const double x = phi[(int64_t)j * ld + s];
        h = (x + kFdScale * fmax(fabs(x), lo)) - x;
      }
      source_tile<MODE, SPECIAL, kEither>(m, smem, arrays, FdIn<MODE>{in, j, lo}, FdOut<FMT>{m, J, dphi, ws, ld, s, j, h});
    }
    __syncthreads();
  }
}

size_t fd_workspace_bytes(int ns, int64_t n) {
  const SourcePlan p = source_plan(ns, n);
  return p.acc_bytes + p.arrays_bytes;
}

template <int MODE, int FMT>
static int launch_fd_t(const DevMech& m, int64_t n, const double* param, const double* phi, int64_t ld, double* J,
                       double* dphi, int* status, double* work, cudaStream_t st) {
  const SourcePlan p = source_plan(m.ns, n);
  auto kern = m.nr_plain < m.nr ? k_fd_jacobian<MODE, FMT, true> : k_fd_jacobian<MODE, FMT, false>;
  int rc;
  if ((rc = set_smem(kern, p.smem))) return rc;
  double* arrays = p.arrays_bytes ? work : nullptr;
  kern<<<p.grid, kSrcWarps * 32, p.smem, st>>>(m, n, param, phi, ld, J, dphi, status,
                                               work + p.arrays_bytes / sizeof(double), arrays);
  return check_cuda(cudaGetLastError(), "k_fd_jacobian launch");
}

int launch_fd_jacobian(const DevMech& m, int mode, int fmt, int64_t n, const double* param, const double* phi,
                       int64_t ld, double* J, double* dphi, int* status, void* work, size_t work_bytes,
                       cudaStream_t st) {
  const size_t need = fd_workspace_bytes(m.ns, n);
  if (!work || work_bytes < need)
    return fail(PJ_ERR_NOMEM, "workspace too small for the finite-difference Jacobian (see pj_workspace_size)");
  double* ws = static_cast<double*>(work);
  if (mode == PJ_CONP) {
    if (fmt == PJ_CSR) return launch_fd_t<PJ_CONP, PJ_CSR>(m, n, param, phi, ld, J, dphi, status, ws, st);
    if (fmt == PJ_CSC) return launch_fd_t<PJ_CONP, PJ_CSC>(m, n, param, phi, ld, J, dphi, status, ws, st);
    return launch_fd_t<PJ_CONP, PJ_DENSE>(m, n, param, phi, ld, J, dphi, status, ws, st);
  }
  if (fmt == PJ_CSR) return launch_fd_t<PJ_CONV, PJ_CSR>(m, n, param, phi, ld, J, dphi, status, ws, st);
  if (fmt == PJ_CSC) return launch_fd_t<PJ_CONV, PJ_CSC>(m, n, param, phi, ld, J, dphi, status, ws, st);
  return launch_fd_t<PJ_CONV, PJ_DENSE>(m, n, param, phi, ld, J, dphi, status, ws, st);
}

}  // namespace pj
