// Differentiation form: vector-Jacobian products of y = (wdot_0 .. wdot_{Ns-1},
// dT/dt) with respect to the state and to the per-reaction Arrhenius
// parameters theta_i = (ln A_i, beta_i, Ea_i) of the high-pressure (or only)
// rate.
//
// Adjoint structure (Sec. 2.2 rates): y depends on the state through the net
// rates q_i and, for dT/dt, through the species energies and the heat
// capacity sum D.  With cotangent u = (u_wdot, u_T),
//   ubar_i = sum_k nu_ki u_k - u_T dE_i / D        (adjoint of q_i)
//   g_Phi  = sum_i ubar_i grad q_i - u_T (delta_jT sum_k Cx_k wdot_k + Tdot grad D) / D
//   g_theta_i = sum_states ubar_i dq_i/dtheta_i,  dq_i/dtheta = (1, ln T, -1/(R_cal T)) Q_i
// with Q_i = q_i for non-falloff reactions and q_i - R_i Pr dc/dPr for falloff
// (k_inf scales R and divides Pr).
//
// The kernel: kVjpWarps warps share a tile of 32 states (lane = state), the
// reactions split among them in a fixed order; FP64-bound like the Jacobian,
// whose short path for plain reactions it shares.  Deterministic for a given
// launch shape: each warp adds its reactions' production rates and amount
// gradients to rows of its own (L2 reductions of one thread to one address
// apply in program order), which are then summed in warp order; the adjoint
// parts ubar_i Q_i of the parameter gradients are written per reaction and
// state and summed over the tile's states with lane = reaction (three FP64
// instructions per 32 reactions and state, where warp shuffles took fifteen
// per reaction), into sums that one lane of the block owns; blocks' sums are
// added in a fixed order.
#include <cuda_runtime.h>

#include <algorithm>

#include "launch.h"
#include "lean_jacobian.cuh"

namespace pj {

constexpr int kVjpWarps = 8;
constexpr int kVjpCtas = 2;

enum VjpSc {
  vT, vV, vP, vInvT, vInvV, vLnT, vLnP, vCtot, vL, vIT, vLP, vCdum, vCxB, vDcpB, vIden, vDdenT, vDdenS, vDCbT, vDCbS,
  vUT, vMRT, vGB, vTv, kVjpSc
};
enum VjpPart { wAcc, wDen, wDden, wNum, wSum, wGT, wGS, wGB, kVjpPart };
enum VjpFlag { xOk, xFast, kVjpFlag };  // xFast: 1 in the fixed point's range; 0: T out of it; 2: some g_k or h_k

__host__ __device__ constexpr size_t vjp_arrays_bytes(int ns) { return (size_t)4 * ns * kTile * sizeof(double); }
__host__ __device__ constexpr size_t vjp_smem_bytes(int ns, bool arrays_smem) {
  return (arrays_smem ? vjp_arrays_bytes(ns) : 0) +
         (size_t)(kVjpSc + kVjpPart * kVjpWarps) * kTile * sizeof(double) + (size_t)kVjpFlag * kTile * sizeof(int);
}

// Per-state values the reaction bodies read, and their accumulators.
struct VjpVars {
  double T, V, P, invT, invV, lnT, lnP, Ctot, dCb_T, dCb_S;
  double uTE;  // u_T R T / D
  FixedState fx;
  double gT, gS, gB;
};

// A plain reaction with at most three factors a side (as lean_jacobian);
// returns ubar Q.
template <int MODE, bool MIXED>
__device__ __forceinline__ double lean_vjp(const DevMech& m, const Rxn* __restrict__ r, const RxnHead& h,
                                           const double* __restrict__ base, VjpVars& v, double* __restrict__ wrow,
                                           double* __restrict__ grow) {
  const int ns = m.ns, bath = ns - 1;
  const double* __restrict__ C = base;
  const double* __restrict__ G = base + ns * kTile;
  const double* __restrict__ H = base + 2 * ns * kTile;
  const double* __restrict__ U = base + 3 * ns * kTile;
  RxnJac a;
  {
    const int4* __restrict__ p = reinterpret_cast<const int4*>(&r->jac);
    int4* q = reinterpret_cast<int4*>(&a);
#pragma unroll
    for (int i = 0; i < 4; i++) q[i] = __ldg(p + i);
  }
  const bool rev = h.rev != 0;
  const LeanK k = lean_constants<MIXED>(m, r, h, G, v.fx, v.lnT, v.invT);
  LeanSide sf, sb;
  double Rn, SV, du;  // SV: V dRn/dV at constant n; du = sum nu u
  lean_shapes(h.code, [&](auto tf, auto tb) {
    constexpr int SF = decltype(tf)::value, SB = decltype(tb)::value;
    constexpr int nfac[5] = {1, 2, 2, 3, 3};
    sf = lean_side<SF>(h.f, C, k.kf);
    sb = lean_side<SB>(h.b, C, k.kr);
    Rn = SB < 0 ? sf.R : sf.R - sb.R;
    constexpr int NF = nfac[SF], NB = SB < 0 ? 0 : nfac[SB < 0 ? 0 : SB];
    SV = 0.0;
    if (MODE == PJ_CONP) {
      if (NF == NB || SB < 0) SV = NF == 1 ? dneg(Rn) : -(double)NF * Rn;
      else SV = (NB == 1 ? sb.R : (double)NB * sb.R) - (NF == 1 ? sf.R : (double)NF * sf.R);
    }
    du = dneg(U[h.f[0]]);
    if (NF > 1) du -= U[h.f[1]];
    if (NF > 2) du -= U[h.f[2]];
    if (SB >= 0) {
      du += U[h.b[0]];
      if (NB > 1) du += U[h.b[1]];
      if (NB > 2) du += U[h.b[2]];
    }
  });
  if (!rev) {
    du += U[h.b[0]];
    if (h.nb > 1) du += U[h.b[1]];
    if (h.nb > 2) du += U[h.b[2]];
  }
  const double de = lean_energy<MIXED>(h, H, h.dnu_i, v.fx.fast);  // sum nu h/RT - dnu
  double dhd = de;
  if (MODE == PJ_CONP && h.dnu_i != 0) dhd = lean_energy<MIXED>(h, H, 0, v.fx.fast);
  const double ub = fma(-v.uTE, dhd, du);
  const double ubV = ub * v.invV;

  // derivatives of the net rate (lean_jacobian)
  const double Ef = fma(a.theta, v.invT, a.beta);
  double qT = fma(sb.R, de, Rn * Ef) * v.invT;
  double qS = MODE == PJ_CONP ? SV * v.invV : 0.0;
  double Gb = 0.0;
  bool has_S = MODE == PJ_CONP;
  if (a.bath) {
    if (a.bath & 1) Gb += sf.d0;
    if (a.bath & 2) Gb += sf.d1;
    if (a.bath & 4) Gb += sf.d2;
    if (a.bath & 8) Gb -= sb.d0;
    if (a.bath & 16) Gb -= sb.d1;
    if (a.bath & 32) Gb -= sb.d2;
    qT = fma(Gb, v.dCb_T, qT);
    if (MODE == PJ_CONP) qS = (a.nbx * sb.R - a.nfx * sf.R) * v.invV;
    qS = fma(Gb, v.dCb_S, qS);
    has_S = true;
  }
  double q = Rn, Q = Rn, ubVc = ubV;
  if (h.kind != PJ_ELEMENTARY) {
    double M = v.Ctot;
    for (int e = __ldg(&r->eff_lo), eh = __ldg(&r->eff_hi); e < eh; e++) {
      if (!PJ_DBG_OK(m.dbg, e >= 0 && e < m.n_eff && __ldg(m.eff_sp + e) >= 0 && __ldg(m.eff_sp + e) < m.ns,
                     PJ_DBG_EFF))
        break;
      M = fma(__ldg(m.eff_am1 + e), C[kTile * __ldg(m.eff_sp + e)], M);
    }
    const double ab = __ldg(&r->alpha_bath);
    const double dMdT = ab * v.dCb_T;
    const double dMdS = MODE == PJ_CONP ? (ab * v.Ctot - M) * v.invV : ab * (v.Ctot / v.P);
    double cT = dMdT, c = M, RcM = Rn;
    if (h.kind != PJ_THIRD_BODY) {
      int64_t l2rk;
      const double rk = lean_falloff<MIXED>(r, k, v.fx, v.lnT, v.invT, l2rk);
      const FalloffC fc =
          falloff_derivatives<MIXED>(r, m.log_tab, h.kind, v.T, v.invT, v.lnT, v.fx.IT, rk, l2rk, M, dMdT);
      c = fc.c;
      cT = fc.cT;
      RcM = Rn * fc.cM;
    }
    q = c * Rn;
    Q = h.kind != PJ_THIRD_BODY ? fma(-RcM, M, q) : q;  // k_inf divides Pr: - Rn Pr dc/dPr
    qT = fma(c, qT, Rn * cT);
    qS = fma(c, qS, RcM * dMdS);
    has_S = true;
    ubVc = ubV * c;
    double Bi = 0.0;
    for (int e = __ldg(&r->eff_lo), eh = __ldg(&r->eff_hi); e < eh; e++) {
      if (!PJ_DBG_OK(m.dbg, e >= 0 && e < m.n_eff, PJ_DBG_EFF)) break;
      const int j = __ldg(m.eff_sp + e);
      const double val = RcM * __ldg(m.eff_am1 + e);
      if (j == bath) Bi -= val;
      else red_add(grow + j * kTile, ubV * val);
    }
    v.gB = fma(ubV, Bi, v.gB);
  }
  if (a.bath) v.gB = fma(-ubVc, Gb, v.gB);
  v.gT = fma(ub, qT, v.gT);
  if (has_S) v.gS = fma(ub, qS, v.gS);

  // production rates and amount gradients into the warp's rows
  const double nq = dneg(q);
#pragma unroll
  for (int s = 0; s < 3; s++) {
    if (s < h.nf) red_add(wrow + h.f[s], nq);
    if (s < h.nb) red_add(wrow + h.b[s], q);
  }
  // slots in species order: the factors last to first (2A + B: A, B)
  auto slot = [&](int sp, double d) { red_add(grow + kTile * sp, ubVc * d); };
  const int nsf = shape_species(a.shape[0]), nsb = rev ? shape_species(a.shape[1]) : 0;
#pragma unroll
  for (int s = 0; s < 3; s++) {
    if (s < nsf && !(a.bath >> s & 1)) slot(__ldg(&r->sp[s]), s == 0 ? sf.d0 : s == 1 ? sf.d1 : sf.d2);
    if (s < nsb && !(a.bath >> (3 + s) & 1))
      slot(__ldg(&r->sp[PJ_MAX_SP + s]), dneg(s == 0 ? sb.d0 : s == 1 ? sb.d1 : sb.d2));
  }
  return ub * Q;
}

// What a reaction needs of its state (sc: this lane's scalars of the tile; ok: a
// valid state), and the sums over a warp's reactions.
__device__ __forceinline__ VjpVars vjp_vars(const double* __restrict__ sc, bool fast, bool ok) {
  auto S = [&](int v) { return sc[v * kTile]; };
  VjpVars v;
  v.T = S(vT);
  v.V = S(vV);
  v.P = S(vP);
  v.invT = S(vInvT);
  v.invV = S(vInvV);
  v.lnT = S(vLnT);
  v.lnP = S(vLnP);
  v.Ctot = S(vCtot);
  v.dCb_T = S(vDCbT);
  v.dCb_S = S(vDCbS);
  v.uTE = ok ? S(vUT) * S(vIden) * (RU * v.T) : 0.0;
  v.fx.L = (uint64_t)__double_as_longlong(S(vL));
  v.fx.IT = (uint64_t)__double_as_longlong(S(vIT));
  v.fx.LP = __double_as_longlong(S(vLP));
  v.fx.fast = fast;
  return v;
}
template <class F>
__device__ __forceinline__ void vjp_sums(VjpVars& v, F&& f) {
  f(0, v.gT);
  f(1, v.gS);
  f(2, v.gB);
}

// Two out-of-line bodies beside the inlined short path.  Both take the state
// from and leave their sums in shared memory (part: this lane's of the warp;
// as general_jacobian), short-path reactions from wGT on and the others from
// wAcc on (free between phases C and E), so that the sums of a state come in the
// same order whichever body its tile needs.
//
// A short-path reaction in a tile with a state outside the fixed point's range,
// each lane by its own state: what a state gives does not depend on its tile
// mates.
template <int MODE>
__device__ __noinline__ static double mixed_vjp(const DevMech& m, double* base, const double* sc, double* part,
                                                const Rxn* __restrict__ r, bool fast, bool ok, double* wrow,
                                                double* grow) {
  part += wGT * kTile;
  VjpVars v = vjp_vars(sc, fast, ok);
  vjp_sums(v, [&](int p, double& x) { x = part[p * kTile]; });
  const double w = lean_vjp<MODE, true>(m, r, load_head(r), base, v, wrow, grow);
  vjp_sums(v, [&](int p, double& x) { part[p * kTile] = x; });
  return w;
}

// Any other reaction at any state.  base: this lane's column of C, g, h, u
// ([4][ns][32]); wrow, grow: the warp's rows of wdot and of d/dn; returns the
// adjoint part of the parameter gradient.
template <int MODE, bool SPECIAL>
__device__ __noinline__ static double general_vjp(const DevMech& m, double* base, const double* sc, double* part,
                                                  const Rxn* __restrict__ r, bool plain, bool fast, bool ok, double* wrow,
                                                  double* grow) {
  enum { aC = 0, aG = 1, aH = 2, aU = 3 };
  part += wAcc * kTile;
  VjpVars v = vjp_vars(sc, fast, ok);
  vjp_sums(v, [&](int p, double& x) { x = part[p * kTile]; });
  StateArrays A;
  A.ns = m.ns;
  A.base = base;
  A.stride = kTile;
  const int bath = m.ns - 1;
  const double T = v.T, P = v.P, invT = v.invT, lnT = v.lnT, invV = v.invV, invT2 = v.invT * v.invT;
  const int kind = __ldg(&r->kind);
  const int nre = __ldg(&r->nreac), npr = __ldg(&r->nprod), rev = __ldg(&r->rev);
  double dlnkf, dlnP, dlnkinf;
  ln_kf_derivatives<SPECIAL>(m, r, kind, lnT, invT, invT2, v.lnP, dlnkf, dlnP, dlnkinf);
  const RateK rk = rate_constants<SPECIAL>(m, A, aG, r, kind, rev, nre, npr, v.fx, lnT, invT, v.lnP);
  double dh = 0.0, du = 0.0;
  for (int a = 0; a < 2 * PJ_MAX_SP; a++) {
    const bool react = a < PJ_MAX_SP;
    if (react ? a >= nre : a - PJ_MAX_SP >= npr) continue;
    const int k = __ldg(&r->sp[a]);
    const double nu = react ? -__ldg(&r->nud[a]) : __ldg(&r->nud[a]);
    const double hk = A.at(aH, k);
    dh = fma(nu, fast ? fixed51_to_double(__double_as_longlong(hk)) : hk, dh);
    du = fma(nu, A.at(aU, k), du);
  }
  double dRf[PJ_MAX_SP], dRr[PJ_MAX_SP];
  const double Rf = side_rate<true>(A, aC, r, 0, __ldg(&r->shape[0]), nre, rk.kf, dRf);
  double Rr = 0.0, dlnkr = 0.0;
  if (rev) {
    Rr = side_rate<true>(A, aC, r, PJ_MAX_SP, __ldg(&r->shape[1]), npr, rk.kr, dRr);
    if (SPECIAL && rev == 2)
      dlnkr = fma(__ldg(m.tab + __ldg(&r->tab_lo) + 2), invT2, __ldg(m.tab + __ldg(&r->tab_lo) + 1) * invT);
    else
      dlnkr = dlnkf - (dh - __ldg(&r->dnu)) * invT;
  }
  const double Rn = Rf - Rr;
  double c = 1.0, dcdT = 0.0, dcdS = 0.0, dcdM = 0.0;
  // d q / d ln k_inf (k_inf: the Arrhenius set the parameter gradient is
  // taken for) = part through the base rate + part through Pr
  double Qpr = 0.0;
  if (has_third_body(kind)) {
    const double M = third_body(m, A, aC, r, v.Ctot);
    const double ab = __ldg(&r->alpha_bath);
    const double dMdT = ab * v.dCb_T;
    const double dMdS = MODE == PJ_CONP ? (ab * v.Ctot - M) * invV : ab * v.Ctot / P;
    if (kind == PJ_THIRD_BODY) {
      c = M;
      dcdM = 1.0;
      dcdT = dMdT;
      dcdS = dMdS;
    } else {
      const double dlnk0 = fma(__ldg(&r->theta0), invT2, __ldg(&r->beta0) * invT);
      double F, FxPr, FT;
      const double Pr = falloff_Pr_F<true>(m, r, kind, v.fx, T, invT, lnT, rk, M, F, FxPr, FT);
      const double i1p = 1.0 / (1.0 + Pr);
      const double dPrdT = Pr * (dlnk0 - dlnkinf) + rk.rk * dMdT;
      double cPr;
      if (SPECIAL && __ldg(&r->chem)) {
        c = F * i1p;
        cPr = i1p * (FxPr / Pr - F * i1p);
        dcdT = i1p * FT + cPr * dPrdT;
      } else {
        const double fr = Pr * i1p;
        c = fr * F;
        cPr = F * i1p * i1p + FxPr * i1p;
        dcdT = fr * FT + cPr * dPrdT;
      }
      dcdM = cPr * rk.rk;
      dcdS = dcdM * dMdS;
      Qpr = -Rn * cPr * Pr;  // k_inf divides Pr
    }
  }
  const double q = c * Rn;
  // the base rate is k_inf unless the reaction is chemically activated or
  // pressure-dependent; with an explicit reverse rate only R' scales
  const bool base_inf = plain || (kind < PJ_PLOG && !__ldg(&r->chem));
  const double Q = (base_inf ? c * ((SPECIAL && rev == 2) ? Rf : Rn) : 0.0) + Qpr;
  double dRdT = Rf * dlnkf - Rr * dlnkr;
  double dRdS = 0.0;
  double Bi = 0.0;
  const double dE = MODE == PJ_CONP ? dh : dh - __ldg(&r->dnu);
  const double ub = fma(-v.uTE, dE, du);
  const double ubV = ub * invV;
  for (int a = 0; a < 2 * PJ_MAX_SP; a++) {
    const bool react = a < PJ_MAX_SP;
    const int b = react ? a : a - PJ_MAX_SP;
    if (react ? b >= nre : b >= npr) continue;
    const int k = __ldg(&r->sp[a]);
    const double nu = react ? -__ldg(&r->nud[a]) : __ldg(&r->nud[a]);
    red_add(wrow + k * kTile, nu * q);
    if (!react && !rev) continue;
    const double d = react ? dRf[b] : -dRr[b];
    if (k == bath) {
      dRdT = fma(d, v.dCb_T, dRdT);
      dRdS = fma(d, v.dCb_S, dRdS);
      Bi -= c * d;
    } else {
      if (MODE == PJ_CONP) dRdS = fma(d, -A.at(aC, k) * invV, dRdS);
      red_add(grow + k * kTile, ubV * (c * d));
    }
  }
  if (SPECIAL && MODE == PJ_CONV && kind >= PJ_PLOG) {
    // P-log / Chebyshev rates depend on P = S; an explicit reverse rate does not
    const double dP = dlnP / P;
    dRdS = fma(Rf, dP, dRdS) - (rev == 1 ? Rr * dP : 0.0);
  }
  v.gT = fma(ub, fma(c, dRdT, Rn * dcdT), v.gT);
  v.gS = fma(ub, fma(c, dRdS, Rn * dcdS), v.gS);
  if (has_third_body(kind)) {
    const double t = Rn * dcdM;
    for (int e = __ldg(&r->eff_lo), eh = __ldg(&r->eff_hi); e < eh; e++) {
      const int j = __ldg(m.eff_sp + e);
      const double val = t * __ldg(m.eff_am1 + e);
      if (j == bath) Bi -= val;
      else red_add(grow + j * kTile, ubV * val);
    }
  }
  v.gB = fma(ubV, Bi, v.gB);
  vjp_sums(v, [&](int p, double& x) { part[p * kTile] = x; });
  return ub * Q;
}

// Workspace of a block: the warps' rows [W][2][ns][32] (wdot, d/dn), ubar Q
// [nr][32], and, unless in shared memory, the arrays [4][ns][32].
__host__ __device__ inline size_t vjp_block_doubles(int ns, int nr, bool arrays_smem) {
  return (size_t)kTile * (2 * kVjpWarps * ns + nr + (arrays_smem ? 0 : 4 * ns));
}

template <int MODE, bool SPECIAL, bool SHARED>
__global__ void __launch_bounds__(kVjpWarps * 32, kVjpCtas)
    k_vjp(const __grid_constant__ DevMech m, int64_t n, const double* __restrict__ param,
          const double* __restrict__ phi, int64_t ld, const double* __restrict__ u_wdot,
          const double* __restrict__ u_T, double* __restrict__ y, double* __restrict__ g_phi,
          double* __restrict__ gth_part, int* status, double* __restrict__ ws) {
  PJ_DYN_SMEM;
  load_exp_table(m.exp_tab);
  const int ns = m.ns, bath = m.ns - 1, nr = m.nr;
  const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  constexpr int W = kVjpWarps;
  ws += (size_t)blockIdx.x * vjp_block_doubles(ns, nr, SHARED);
  double* const rows = ws + lane;                                         // [W][2][ns][32]
  double* const wq = ws + (size_t)2 * W * ns * kTile;                     // [nr][32]
  double* const base = SHARED ? smem + lane : wq + (size_t)nr * kTile + lane;  // C, g, h, u: [4][ns][32]
  double* const tsm = SHARED ? smem + 4 * ns * kTile : smem;
  double* const sc = tsm + lane;
  double* const part = tsm + kVjpSc * kTile + lane;
  int* const flags = reinterpret_cast<int*>(tsm + (kVjpSc + kVjpPart * W) * kTile) + lane;
  double* const my_part = gth_part + (size_t)blockIdx.x * nr * 3;
  double* const C = base;
  double* const G = base + ns * kTile;
  double* const H = base + 2 * ns * kTile;
  double* const U = base + 3 * ns * kTile;
  auto S = [&](int i) -> double& { return sc[i * kTile]; };
  auto Pw = [&](int w, int i) -> double& { return part[(w * kVjpPart + i) * kTile]; };
  auto sum_parts = [&](int i) {
    double t = 0.0;
    for (int w = 0; w < W; w++) t += Pw(w, i);
    return t;
  };
  auto sum_rows = [&](int which, int k) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < W; w++) t += __ldcg(rows + ((size_t)(2 * w + which) * ns + k) * kTile);
    return t;
  };

  for (int64_t tile = blockIdx.x; tile * kTile < n; tile += gridDim.x) {
    const int64_t s = tile * kTile + lane;
    const bool act = s < n;
    double* const wrow = rows + (size_t)(2 * warp) * ns * kTile;
    double* const grow = wrow + (size_t)ns * kTile;

    // A: the state's scalars (warp 0; a lane without a valid T, V, P takes a
    // dummy state); zero the warp's rows
    if (warp == 0) {
      double T = 1000.0, V = 1.0, P = 1e5, uT = 0.0;
      bool ok0 = false;
      if (act) {
        const double T_ = phi[s], S_ = phi[ld + s], par = param[s];
        const double V_ = MODE == PJ_CONP ? S_ : par, P_ = MODE == PJ_CONP ? par : S_;
        ok0 = (T_ > 0.0) && (V_ > 0.0) && (P_ > 0.0) && isfinite(T_) && isfinite(V_) && isfinite(P_);
        if (ok0) {
          T = T_;
          V = V_;
          P = P_;
          uT = u_T[s];
        }
      }
      const double invT = 1.0 / T;
      double lnT;
      FixedState fx;
      temperature_terms(m, T, invT, lnT, fx);
      const double Ctot = P / (RU * T);
      S(vT) = T;
      S(vV) = V;
      S(vP) = P;
      S(vInvT) = invT;
      S(vInvV) = 1.0 / V;
      S(vLnT) = lnT;
      S(vLnP) = m.has_pdep ? log(P) : 0.0;
      S(vCtot) = Ctot;
      S(vL) = __longlong_as_double((long long)fx.L);
      S(vIT) = __longlong_as_double((long long)fx.IT);
      S(vLP) = __longlong_as_double((long long)fx.LP);
      S(vCdum) = Ctot / ns;
      S(vUT) = uT;
      S(vMRT) = -1.0 / (R_CAL * T);
      flags[xOk * kTile] = ok0;
      flags[xFast * kTile] = fx.fast;
    }
    for (int k = 0; k < 2 * ns; k++) wrow[k * kTile] = 0.0;
    __syncthreads();

    // B: concentrations, thermo and cotangents of the warp's species
    {
      const double T = S(vT), V = S(vV), invT = S(vInvT), invV = S(vInvV), lnT = S(vLnT), cdum = S(vCdum);
      const bool ok0 = flags[xOk * kTile] != 0;
      double acc = 0.0, den = 0.0, dden = 0.0;
      const bool fast0 = flags[xFast * kTile] != 0;
      bool fast = fast0;
      for (int k = warp; k < ns; k += W) {
        const double* cb = nasa_block(m, k, T);
        double cp, g, cp2, dcp;
        nasa_cp_g(cb, T, invT, lnT, cp, g);
        nasa_cp(cb, T, cp2, dcp);
        G[k * kTile] = gibbs_entry(m, g, fast);
        H[k * kTile] = enthalpy_entry(m, nasa_h(cb, T, invT), fast);
        U[k * kTile] = ok0 ? u_wdot[(int64_t)k * ld + s] : 0.0;
        const double cx = MODE == PJ_CONP ? cp : cp - 1.0;
        if (k < bath) {
          const double c = ok0 ? concentration(phi[(int64_t)(k + 2) * ld + s], V, invV) : cdum;
          C[k * kTile] = c;
          acc += c;
          den = fma(c, cx, den);
          dden = fma(c, dcp, dden);
        } else {
          S(vCxB) = cx;
          S(vDcpB) = dcp;
        }
      }
      if (fast0 && !fast) flags[xFast * kTile] = 2;  // found out of range part of the way
      Pw(warp, wAcc) = acc;
      Pw(warp, wDen) = den;
      Pw(warp, wDden) = dden;
    }
    __syncthreads();

    // C: bath gas by subtraction, validity (an invalid state's cotangents
    // become zero), the energy equation's denominator and its derivatives; the
    // entries of a state found out of range, again
    if (flags[xFast * kTile] == 2) {
      const double T = S(vT), invT = S(vInvT), lnT = S(vLnT);
      for (int k = warp; k < ns; k += W) {
        const double* cb = nasa_block(m, k, T);
        double cp, g;
        nasa_cp_g(cb, T, invT, lnT, cp, g);
        G[k * kTile] = g;
        H[k * kTile] = nasa_h(cb, T, invT);
      }
    }
    if (warp == 0) {
      const double Ctot = S(vCtot), P = S(vP), invT = S(vInvT), invV = S(vInvV);
      const double acc = sum_parts(wAcc);
      const double Cns = Ctot - acc;
      const bool ok = flags[xOk * kTile] != 0 && isfinite(acc) && isfinite(Cns) && !(Cns < -1e-12 * Ctot);
      C[bath * kTile] = Cns;
      const double den = RU * (sum_parts(wDen) + Cns * S(vCxB));
      const double Cx_bath = RU * S(vCxB);
      const double dCb_T = -Ctot * invT;
      const double dCb_S = MODE == PJ_CONP ? (Ctot - Cns) * invV : Ctot / P;
      S(vIden) = 1.0 / den;
      S(vDCbT) = dCb_T;
      S(vDCbS) = dCb_S;
      S(vDdenT) = RU * (sum_parts(wDden) + Cns * S(vDcpB)) + Cx_bath * dCb_T;
      S(vDdenS) = MODE == PJ_CONP ? (Cx_bath * Ctot - den) * invV : Cx_bath * Ctot / P;
      flags[xOk * kTile] = ok;
      if (!ok) S(vMRT) = 0.0;  // -1/T may be infinite; the state takes no part in the parameters' sums
      if (act && !ok) {
        write_nan_state(g_phi, ld, s, ns + 1);
        write_nan_state(y, ld, s, ns + 1);
        if (status) atomicAdd(status, 1);
      }
    }
    __syncthreads();
    const bool ok = flags[xOk * kTile] != 0;
    const bool fast = flags[xFast * kTile] == 1;
    const bool fast_tile = __all_sync(0xffffffffu, fast);  // the same in every warp

    // D: the warp's reactions, in a fixed order
    {
      double* const my_sums = part + warp * kVjpPart * kTile;
      VjpVars v = vjp_vars(sc, true, ok);
      vjp_sums(v, [&](int p, double& x) { x = my_sums[(wAcc + p) * kTile] = my_sums[(wGT + p) * kTile] = 0.0; });
      for (int i = warp; i < nr; i += W) {
        const Rxn* __restrict__ r = m.rxn + i;
        const RxnHead h = load_head(r);
        double w;
        if (fast_tile && h.lean) w = lean_vjp<MODE, false>(m, r, h, base, v, wrow, grow);
        else if (h.lean) w = mixed_vjp<MODE>(m, base, sc, my_sums, r, fast, ok, wrow, grow);
        else w = general_vjp<MODE, SPECIAL>(m, base, sc, my_sums, r, i < m.nr_plain, fast, ok, wrow, grow);
        wq[(size_t)i * kTile + lane] = ok ? w : 0.0;
      }
      vjp_sums(v, [&](int p, double& x) {
        my_sums[(wGT + p) * kTile] = (my_sums[(wGT + p) * kTile] + x) + my_sums[(wAcc + p) * kTile];
      });
    }
    __syncthreads();

    // E: the warp's species (G becomes Cx_k); then, lane = reaction, the
    // parameter gradients of the tile
    {
      const double T = S(vT);
      double num = 0.0, sumCxW = 0.0;
      for (int k = warp; k < ns; k += W) {
        double cp, dcp;
        nasa_cp(nasa_block(m, k, T), T, cp, dcp);
        const double cx = RU * (MODE == PJ_CONP ? cp : cp - 1.0);
        const double hk = fast ? fixed51_to_double(__double_as_longlong(H[k * kTile])) : H[k * kTile];
        const double wk = sum_rows(0, k);
        G[k * kTile] = cx;
        num = fma(MODE == PJ_CONP ? hk : hk - 1.0, wk, num);
        sumCxW = fma(cx, wk, sumCxW);
        if (ok) y[(int64_t)k * ld + s] = wk;
      }
      Pw(warp, wNum) = num;
      Pw(warp, wSum) = sumCxW;
      for (int i = warp * 32 + lane; i < nr; i += W * 32) {
        const double2* __restrict__ q = reinterpret_cast<const double2*>(wq + (size_t)i * kTile);
        double s0 = 0.0, s1 = 0.0, s2 = 0.0;
        for (int t = 0; t < kTile / 2; t++) {
          const double2 x = __ldcg(q + t);
          s0 += x.x;
          s1 = fma(x.x, tsm[vLnT * kTile + 2 * t], s1);
          s2 = fma(x.x, tsm[vMRT * kTile + 2 * t], s2);
          s0 += x.y;
          s1 = fma(x.y, tsm[vLnT * kTile + 2 * t + 1], s1);
          s2 = fma(x.y, tsm[vMRT * kTile + 2 * t + 1], s2);
        }
        double* p = my_part + (size_t)i * 3;
        if (tile != (int64_t)blockIdx.x) {
          s0 += p[0];
          s1 += p[1];
          s2 += p[2];
        }
        p[0] = s0;
        p[1] = s1;
        p[2] = s2;
      }
    }
    __syncthreads();

    // F: dT/dt and the gradients in T and S (warp 0)
    if (warp == 0) {
      const double T = S(vT), iden = S(vIden), uT = ok ? S(vUT) : 0.0;
      const double Tdot = -(sum_parts(wNum) * (RU * T)) * iden;
      S(vGB) = sum_parts(wGB);
      S(vTv) = uT * Tdot * S(vInvV) * iden;
      if (ok) {
        y[(int64_t)ns * ld + s] = Tdot;
        g_phi[s] = sum_parts(wGT) + uT * (-(sum_parts(wSum) + Tdot * S(vDdenT)) * iden);
        g_phi[ld + s] = sum_parts(wGS) + uT * (-(Tdot * S(vDdenS)) * iden);
      }
    }
    __syncthreads();

    // G: the amount gradients
    {
      const double gB = S(vGB), tv = S(vTv), Cxb = G[bath * kTile];
      for (int j = warp; j < bath; j += W) {
        const double acc = sum_rows(1, j);
        if (ok) g_phi[(int64_t)(j + 2) * ld + s] = acc + gB - tv * (G[j * kTile] - Cxb);
      }
    }
    __syncthreads();
  }
}

// g_theta[perm[i]][p]: the blocks' sums, 32 interleaved partial sums (lane =
// block modulo 32) added by a fixed tree.
__global__ void __launch_bounds__(128) k_vjp_reduce(int nr, int blocks, const double* __restrict__ part,
                                                    const int32_t* __restrict__ perm, double* __restrict__ g_theta) {
  const int lane = threadIdx.x & 31;
  const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (t >= (int64_t)nr * 3) return;
  double acc = 0.0;
  for (int b = lane; b < blocks; b += 32) acc += part[(int64_t)b * nr * 3 + t];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) g_theta[(int64_t)perm[t / 3] * 3 + t % 3] = acc;
}

// ---------------------------------------------------------------------------
// launch
// ---------------------------------------------------------------------------
struct VjpPlan {
  bool arrays_smem;
  int grid;
  size_t smem, block_bytes, part_bytes;
};

// arrays in shared memory where a block's fit; the grid: as many blocks as
// are resident
static VjpPlan vjp_plan(const DevMech& m, int64_t n) {
  VjpPlan p{};
  p.arrays_smem = vjp_smem_bytes(m.ns, true) <= kSmemCap;
  p.smem = vjp_smem_bytes(m.ns, p.arrays_smem);
  const int ctas = p.smem + kBlockOverhead <= kSmemPerSm / kVjpCtas ? kVjpCtas : 1;
  const int64_t tiles = (n + kTile - 1) / kTile;
  p.grid = (int)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)sm_count() * ctas));
  p.block_bytes = vjp_block_doubles(m.ns, m.nr, p.arrays_smem) * sizeof(double);
  p.part_bytes = (size_t)p.grid * m.nr * 3 * sizeof(double);
  return p;
}

size_t form_workspace_bytes(int op, const DevMech& m, int64_t n) {
  if (op == PJ_OP_VJP) {
    const VjpPlan p = vjp_plan(m, n);
    return p.block_bytes * p.grid + p.part_bytes + 15;  // the kernel reads 16-byte vectors
  }
  return source_plan(m.ns, n).arrays_bytes;
}

int launch_vjp(const DevMech& m, int mode, int64_t n, const double* param, const double* phi, int64_t ld,
               const double* u_wdot, const double* u_T, double* y, double* g_phi, double* g_theta, int* status,
               void* work, size_t work_bytes, cudaStream_t st) {
  const VjpPlan p = vjp_plan(m, n);
  if (!work || work_bytes < p.block_bytes * p.grid + p.part_bytes + 15)
    return fail(PJ_ERR_NOMEM, "workspace too small for pj_vjp (see pj_workspace_size)");
  char* const aligned = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(work) + 15) & ~uintptr_t(15));
  double* ws = reinterpret_cast<double*>(aligned);
  double* part = reinterpret_cast<double*>(aligned + p.block_bytes * p.grid);
  const bool special = m.nr_plain < m.nr;
  auto pick = [&](auto shared) {
    constexpr bool SH = decltype(shared)::value;
    return mode == PJ_CONP ? (special ? k_vjp<PJ_CONP, true, SH> : k_vjp<PJ_CONP, false, SH>)
                           : (special ? k_vjp<PJ_CONV, true, SH> : k_vjp<PJ_CONV, false, SH>);
  };
  auto kern = p.arrays_smem ? pick(BoolTag<true>{}) : pick(BoolTag<false>{});
  int rc;
  if ((rc = set_smem(kern, p.smem))) return rc;
  kern<<<p.grid, kVjpWarps * 32, p.smem, st>>>(m, n, param, phi, ld, u_wdot, u_T, y, g_phi, part, status, ws);
  if ((rc = check_cuda(cudaGetLastError(), "k_vjp launch"))) return rc;
  const int64_t nt = (int64_t)m.nr * 3;
  if (nt > 0) {
    k_vjp_reduce<<<(unsigned)((nt + 3) / 4), 128, 0, st>>>(m.nr, p.grid, part, m.perm, g_theta);
    if ((rc = check_cuda(cudaGetLastError(), "k_vjp_reduce launch"))) return rc;
  }
  return PJ_OK;
}

}  // namespace pj
