// Device helpers shared by the kernels of kinetics.cu and forms.cu: state
// loading, falloff broadening, reaction-side products, rate constants, third
// bodies, production-rate scatter and reductions.
#pragma once

#include <cuda_runtime.h>

#include "kinetics_device.cuh"

#ifndef PJ_DYN_SMEM
#define PJ_DYN_SMEM extern __shared__ double smem[]
#endif

namespace pj {

// Per-state inputs of the fixed-point rate constants (fixed_math.cuh).  fast:
// they may be used (128 K <= T < 65536 K and every |g_k/RT| in range, see
// gibbs_entry); other states take the FP64 path (rate_constants_fp64), out of
// line.
struct FixedState {
  uint64_t L, IT;  // log2(T) 2^59, 2^70 / T
  int64_t LP;      // log2(P_std / (R T)) 2^51
  bool fast;
};

struct StateScalars {
  double T, V, P, invT, lnT, Ctot;
  double lnP;  // ln P [Pa], formed only when some reaction depends on pressure
  FixedState fx;
};

// ln T and the fixed-point inputs of temperature T > 0 (invT = 1/T rounded).
// 1/T carries the residual of the rounding, ln T is log2(T) ln 2 from the
// fixed point: both at least as exact as the FP64 operations.
__device__ __forceinline__ void temperature_terms(const DevMech& m, double T, double invT, double& lnT,
                                                  FixedState& f) {
  f.fast = T >= 128.0 && T < 65536.0;
  f.L = f.IT = 0;
  f.LP = 0;
  if (!f.fast) {
    lnT = log(T);
    return;
  }
  int e;
  const uint64_t l = log2_fixed((uint64_t)__double_as_longlong(T), e, m.log_tab);
  f.L = ((uint64_t)e << 59) + (l >> 3);
  f.LP = m.log2_pstd_fx - (int64_t)(f.L >> 8);
  lnT = __longlong_as_double((long long)fixed_to_double((int64_t)mulhi_approx(f.L, 0xb17217f7d1cf79acull), 59));
  f.IT = __double2ull_rn(invT * 0x1p70) + (uint64_t)__double2ll_rn(fma(-T, invT, 1.0) * (invT * 0x1p70));
}

// What the reactions read of g_k/RT: log2 units 2^51 at a state within the
// fixed point's range, else the value itself.  Clears fast when g is out of
// range; entries made before that have to be made again.
__device__ __forceinline__ double gibbs_entry(const DevMech& m, double g, bool& fast) {
  fast = fast && ((uint32_t)__double2hiint(g) & 0x7fffffffu) < m.fx_g_hi;
  return fast ? __longlong_as_double(__double2ll_rn(g * (1.4426950408889634074 * 0x1p51))) : g;
}

// The same of h_k/RT: units 2^51.
__device__ __forceinline__ double enthalpy_entry(const DevMech& m, double h, bool& fast) {
  fast = fast && ((uint32_t)__double2hiint(h) & 0x7fffffffu) < m.fx_h_hi;
  return fast ? __longlong_as_double(__double2ll_rn(h * 0x1p51)) : h;
}

// g_k/RT of every species as it is: a state that was found out of range part
// of the way.  Out of line.
template <class SA>
__device__ __noinline__ static void gibbs_entries_again(const DevMech& m, const SA A, int aG, double T, double invT,
                                                        double lnT) {
  for (int k = 0; k < m.ns; k++) {
    double cp, g;
    nasa_cp_g(nasa_block(m, k, T), T, invT, lnT, cp, g);
    A.at(aG, k) = g;
  }
}

// 2^(y 2^-51) as a double
__device__ __forceinline__ double exp2_51(int64_t y) {
  return __longlong_as_double(
      (long long)pack_double_any((int)(y >> 51), exp2_significand((uint64_t)y << 13, pj_exp_tab)));
}

// log2 of a positive normal double, 2^51; ok = false for anything else
__device__ __forceinline__ int64_t log2_51(const LogEntry* __restrict__ log_tab, double x, bool& ok) {
  ok = ok && (uint32_t)__double2hiint(x) - 0x00100000u < 0x7fe00000u;
  int e;
  const uint64_t l = log2_fixed((uint64_t)__double_as_longlong(x), e, log_tab);
  return ((int64_t)e << 51) + (int64_t)(l >> 11);
}

// y 2^-51
__device__ __forceinline__ double fixed51_to_double(int64_t y) {
  return __longlong_as_double((long long)fixed_to_double(y, 51));
}

// n / V from iV = 1/V rounded: one correction of the quotient's residual, so
// that it rounds as the division does but for rare halfway cases (three FP64
// instructions for about nine).
__device__ __forceinline__ double concentration(double n, double V, double iV) {
  if ((uint32_t)__double2hiint(V) - 0x01800000u >= 0x7c000000u) return n / V;  // 1/V would leave the normal range
  const double c = n * iV;
  return fma(fma(-c, V, n), iV, c);
}

__device__ __forceinline__ bool has_third_body(int kind) { return kind >= PJ_THIRD_BODY && kind <= PJ_SRI; }

// Load one state, fill C_k (k < Ns-1 as n_k/V; the bath gas as C_tot minus
// the others summed in species order) and check validity.
template <int MODE, class SA>
__device__ __forceinline__ bool load_state(const DevMech& m, const double* __restrict__ phi,
                                           const double* __restrict__ param, int64_t ld, int64_t s,
                                           const SA& A, int aC, StateScalars& st) {
  const int ns = m.ns;
  const double T = phi[s], S = phi[ld + s], par = param[s];
  const double V = MODE == PJ_CONP ? S : par;
  const double P = MODE == PJ_CONP ? par : S;
  bool ok = (T > 0.0) && (V > 0.0) && (P > 0.0) && isfinite(T) && isfinite(V) && isfinite(P);
  double acc = 0.0;
  const double iV = 1.0 / V;
  for (int k = 0; k < ns - 1; k++) {
    const double c = concentration(phi[(int64_t)(k + 2) * ld + s], V, iV);
    A.at(aC, k) = c;
    acc += c;
  }
  const double Ctot = P / (RU * T);
  st.lnP = m.has_pdep ? log(P) : 0.0;
  const double Cns = Ctot - acc;
  A.at(aC, ns - 1) = Cns;
  ok = ok && isfinite(acc) && isfinite(Cns) && !(Cns < -1e-12 * Ctot);
  st.T = T;
  st.V = V;
  st.P = P;
  st.invT = 1.0 / T;
  temperature_terms(m, T, st.invT, st.lnT, st.fx);
  st.Ctot = Ctot;
  return ok;
}

// 1/x for x well within the normal range: the hardware's approximation and
// two Newton steps (four FMAs; an IEEE division issues about nine FP64
// instructions).
__device__ __forceinline__ double reciprocal(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

// 1 / (1 + Pr); Pr beyond 2^1000 (or not finite, or negative) by division
__device__ __forceinline__ double inverse_1p(double Pr) {
  if ((uint32_t)__double2hiint(Pr) >= 0x7e700000u) return 1.0 / (1.0 + Pr);
  return reciprocal(1.0 + Pr);
}

// Troe / SRI broadening factor F(T, Pr).  With derivatives also returns FxPr
// = Pr dF/dPr (at fixed T) and FT = dF/dT (at fixed Pr).  fxr: which of Troe's
// exponents fit the fixed point (Rxn::troe_fx; the third also needs 128 <= T,
// IT = 2^70 / T); l2Pr = log2(Pr) 2^51; ok = false, with nothing returned, when
// F_cent (or Z) is not a positive normal number.
//
// Troe: with D = N - 0.14 xc and S = D^2 + xc^2, log10 F = L g, g = D^2 / S
// (1 / (1 + (xc/D)^2)), so that F and its derivatives take one reciprocal:
// dg/dx = -2 N xc D / S^2.  Exponents, exponentials and logarithms are fixed
// point: a falloff reaction's 126 FP64 instructions were 22 % of the
// 53-species Jacobian's and 45 % of its source terms'.
template <bool DERIV>
__device__ __forceinline__ double falloff_F(const LogEntry* __restrict__ log_tab, const Rxn* __restrict__ r, int kind,
                                            double T, double invT, double lnT, uint64_t IT, int fxr, int64_t l2Pr,
                                            bool& ok,
                                            double& FxPr, double& FT) {
  FxPr = 0.0;
  FT = 0.0;
  constexpr double LOG10_2 = 0.30102999566398119521;
  if (kind == PJ_TROE) {
    const double a = __ldg(&r->fp[0]), iT3 = __ldg(&r->fp[1]), iT1 = __ldg(&r->fp[2]);
    const double T2 = __ldg(&r->fp[3]);
    const uint64_t tb = (uint64_t)__double_as_longlong(T);
    const uint64_t X = ((tb << 11) | 0x8000000000000000ull) >> (1039 - (int)(tb >> 52));  // T 2^47
    const double e3 = fxr & 1 ? exp2_51(-(int64_t)mulhi_approx(__ldg(&r->tT3), X)) : pj_exp(-T * iT3);
    const double e1 = fxr & 2 ? exp2_51(-(int64_t)mulhi_approx(__ldg(&r->tT1), X)) : pj_exp(-T * iT1);
    double e2 = 0.0;
    if (fxr & 4) e2 = exp2_51(-(int64_t)mulhi_approx(__ldg(&r->tT2), IT));
    else if (__ldg(&r->fp[4]) != 0.0) e2 = pj_exp(-T2 * invT);
    const double Fcent = fma(1.0 - a, e3, fma(a, e1, e2));
    const int64_t l2F = log2_51(log_tab, Fcent, ok);
    if (!ok) return 1.0;
    const double L = fixed51_to_double(l2F) * LOG10_2;
    const double xc = fma(fixed51_to_double(l2Pr), LOG10_2, fma(-0.67, L, -0.4));
    const double NN = fma(-1.27, L, 0.75);
    const double D = fma(-0.14, xc, NN);
    const double D2 = D * D;
    const double iS = reciprocal(fma(xc, xc, D2));
    const double g = D2 * iS;
    // F = 2^(l2F g): the product in fixed point while |log2 F_cent| < 16
    const uint64_t gb = (uint64_t)__double_as_longlong(g);
    const int gs = 1023 - (int)(gb >> 52);
    double F;
    if ((uint64_t)(l2F + (1ll << 55)) < (1ull << 56) && gs >= 0 && gs < 64)
      F = exp2_51((mulhi_su(l2F << 8, ((gb << 11) | 0x8000000000000000ull) >> gs) + 64) >> 7);
    else
      F = pj_exp(LN10 * (L * g));
    if (DERIV) {
      const double Li = L * iS;
      const double t = -2.0 * (xc * D) * (Li * iS);  // L dg/dx / N
      const double dlg_dL = fma(t, fma(1.1762, xc, -0.67 * D), g);
      const double dFcent = fma(T2 * (invT * invT), e2, -fma((1.0 - a) * iT3, e3, (a * iT1) * e1));
      FxPr = F * (t * NN);
      FT = F * dlg_dL * (dFcent * reciprocal(Fcent));
    }
    return F;
  }
  if (kind == PJ_SRI) {
    const double a = __ldg(&r->fp[0]), b = __ldg(&r->fp[1]), ic = __ldg(&r->fp[2]);
    const double d = __ldg(&r->fp[3]), e = __ldg(&r->fp[4]);
    const double x = fixed51_to_double(l2Pr) * LOG10_2;
    const double X = reciprocal(fma(x, x, 1.0));
    const double eb = pj_exp(-b * invT), ec = pj_exp(-T * ic);
    const double Z = a * eb + ec;
    const double lnZ = fixed51_to_double(log2_51(log_tab, Z, ok)) * 0.69314718055994530942;
    if (!ok) return 1.0;
    const double F = d * pj_exp(X * lnZ + e * lnT);
    if (DERIV) {
      FxPr = F * (lnZ * (-2.0 * x * X * X)) * (1.0 / LN10);
      const double dZ = (a * b) * invT * invT * eb - ic * ec;
      FT = F * (X * dZ / Z + e * invT);
    }
    return F;
  }
  return 1.0;  // Lindemann
}

// The same with the library's logarithm, for any Pr and F_cent (zero, subnormal,
// negative or not finite).  Out of line.
__device__ __noinline__ static double falloff_F_library(const Rxn* __restrict__ r, int kind, double T, double invT,
                                                        double lnT, double Pr, double& FxPr, double& FT) {
  FxPr = 0.0;
  FT = 0.0;
  if (kind == PJ_TROE) {
    const double a = __ldg(&r->fp[0]), iT3 = __ldg(&r->fp[1]), iT1 = __ldg(&r->fp[2]);
    const double T2 = __ldg(&r->fp[3]), has2 = __ldg(&r->fp[4]);
    const double e3 = exp(-T * iT3), e1 = exp(-T * iT1);
    const double e2 = has2 != 0.0 ? exp(-T2 * invT) : 0.0;
    const double Fcent = (1.0 - a) * e3 + a * e1 + e2;
    const double L = log10(Fcent);
    const double x = log10(Pr);
    const double cc = -0.4 - 0.67 * L;
    const double NN = 0.75 - 1.27 * L;
    const double xc = x + cc;
    const double D = NN - 0.14 * xc;
    const double f1 = xc / D;
    const double g = 1.0 / (1.0 + f1 * f1);
    const double F = exp(LN10 * (L * g));
    const double iD2 = 1.0 / (D * D);
    const double m2fg2 = -2.0 * f1 * g * g;
    const double dlg_dL = g + L * m2fg2 * (-0.67 * D + 1.1762 * xc) * iD2;
    const double dFcent = -(1.0 - a) * iT3 * e3 - a * iT1 * e1 + T2 * (invT * invT) * e2;
    FxPr = F * (L * m2fg2 * NN * iD2);
    FT = F * dlg_dL * dFcent / Fcent;
    return F;
  }
  if (kind == PJ_SRI) {
    const double a = __ldg(&r->fp[0]), b = __ldg(&r->fp[1]), ic = __ldg(&r->fp[2]);
    const double d = __ldg(&r->fp[3]), e = __ldg(&r->fp[4]);
    const double x = log10(Pr);
    const double X = 1.0 / (1.0 + x * x);
    const double eb = exp(-b * invT), ec = exp(-T * ic);
    const double Z = a * eb + ec;
    const double lnZ = log(Z);
    const double F = d * exp(X * lnZ + e * lnT);
    FxPr = F * (lnZ * (-2.0 * x * X * X)) * (1.0 / LN10);
    const double dZ = (a * b) * invT * invT * eb - ic * ec;
    FT = F * (X * dZ / Z + e * invT);
    return F;
  }
  return 1.0;
}

__device__ __forceinline__ double dneg(double x) {
  return __longlong_as_double(__double_as_longlong(x) ^ (long long)0x8000000000000000ULL);
}

// nu * x with the common nu = +-1 done as a sign flip (integer pipe)
__device__ __forceinline__ double nu_times(int nu, double nud, double x) {
  if (nu == 1) return x;
  if (nu == -1) return dneg(x);
  return nud * x;
}

// R = k * prod_a C_a^nu_a over one reaction side (positions off .. off+n-1)
// and, with DER, dR[a] = dR/dC_a.  The shape code selects the minimal
// multiply sequence; SH_GEN falls back to a general product.
template <bool DER, class SA>
__device__ __forceinline__ double side_rate(const SA& A, int aC, const Rxn* __restrict__ r, int off,
                                            int shape, int n, double k, double (&dR)[PJ_MAX_SP]) {
  switch (shape) {
    case SH_1: {
      const double c0 = A.at(aC, __ldg(&r->sp[off]));
      if (DER) dR[0] = k;
      return k * c0;
    }
    case SH_2: {
      const double c0 = A.at(aC, __ldg(&r->sp[off]));
      const double t = k * c0;
      if (DER) dR[0] = t + t;
      return t * c0;
    }
    case SH_11: {
      const double c0 = A.at(aC, __ldg(&r->sp[off])), c1 = A.at(aC, __ldg(&r->sp[off + 1]));
      const double t = k * c1;
      if (DER) {
        dR[0] = t;
        dR[1] = k * c0;
      }
      return t * c0;
    }
    case SH_21: {
      const double c0 = A.at(aC, __ldg(&r->sp[off])), c1 = A.at(aC, __ldg(&r->sp[off + 1]));
      const double t = k * c0;
      const double t1 = t * c1;
      if (DER) {
        dR[0] = t1 + t1;
        dR[1] = t * c0;
      }
      return t1 * c0;
    }
    case SH_111: {
      const double c0 = A.at(aC, __ldg(&r->sp[off])), c1 = A.at(aC, __ldg(&r->sp[off + 1]));
      const double c2 = A.at(aC, __ldg(&r->sp[off + 2]));
      const double t2 = k * c2;
      const double t12 = t2 * c1;
      if (DER) {
        dR[0] = t12;
        dR[1] = t2 * c0;
        dR[2] = (k * c0) * c1;
      }
      return t12 * c0;
    }
    default: {
      double pw[PJ_MAX_SP], dpw[PJ_MAX_SP];
#pragma unroll
      for (int a = 0; a < PJ_MAX_SP; a++) {
        pw[a] = 1.0;
        dpw[a] = 0.0;
        if (a < n) {
          const int v = __ldg(&r->nu[off + a]);
          const double c = A.at(aC, __ldg(&r->sp[off + a]));
          const double cm = powi(c, v - 1);
          pw[a] = cm * c;
          dpw[a] = v * cm;
        }
      }
      double R = k;
#pragma unroll
      for (int a = 0; a < PJ_MAX_SP; a++)
        if (a < n) R *= pw[a];
      if (DER) {
#pragma unroll
        for (int a = 0; a < PJ_MAX_SP; a++) {
          if (a >= n) continue;
          double p = k * dpw[a];
#pragma unroll
          for (int b = 0; b < PJ_MAX_SP; b++)
            if (b != a && b < n) p *= pw[b];
          dR[a] = p;
        }
      }
      return R;
    }
  }
}

// ln k of a P-log or Chebyshev reaction and, with DER, d ln k / dT and
// d ln k / d ln P.  P-log: Arrhenius rates at ascending ln P_m (table rows
// ln P, ln A, beta, theta), ln k linear in ln P on [ln P_m, ln P_m+1), held at
// the end values below the first and from the last pressure on.  Chebyshev:
// ln k = sum_t sum_p (ln10 a_tp) phi_t(T~) phi_p(P~) with T~ = cT1/T + cT0,
// P~ = cP1 ln P + cP0 and phi_n the Chebyshev polynomials (three-term
// recurrence, which also extends them outside [-1, 1]).
// Not inlined: it runs only for pressure-dependent reactions, and keeping it
// out of the reaction loop keeps that loop's register allocation unchanged.
template <bool DER>
__device__ __noinline__ double lnk_pdep(const DevMech& m, const Rxn* __restrict__ r, int kind, double lnT,
                                        double invT, double lnP, double& d_T, double& d_lnP) {
  const double* __restrict__ t = m.tab + __ldg(&r->tab_lo) + (__ldg(&r->rev) == 2 ? 3 : 0);
  if (kind == PJ_PLOG) {
    const int n = __ldg(&r->tab_n);
    auto lnk_at = [&](int j) { return fma(__ldg(t + 4 * j + 2), lnT, __ldg(t + 4 * j + 1)) - __ldg(t + 4 * j + 3) * invT; };
    auto dT_at = [&](int j) { return fma(__ldg(t + 4 * j + 3), invT * invT, __ldg(t + 4 * j + 2) * invT); };
    if (lnP < __ldg(t) || n == 1) {
      if (DER) { d_T = dT_at(0); d_lnP = 0.0; }
      return lnk_at(0);
    }
    if (lnP >= __ldg(t + 4 * (n - 1))) {
      if (DER) { d_T = dT_at(n - 1); d_lnP = 0.0; }
      return lnk_at(n - 1);
    }
    int j = 0;
    while (j + 2 < n && lnP >= __ldg(t + 4 * (j + 1))) j++;
    const double p0 = __ldg(t + 4 * j), p1 = __ldg(t + 4 * (j + 1));
    const double k0 = lnk_at(j), k1 = lnk_at(j + 1);
    const double slope = (k1 - k0) / (p1 - p0);
    if (DER) {
      const double w = (lnP - p0) / (p1 - p0);
      d_T = fma(w, dT_at(j + 1) - dT_at(j), dT_at(j));
      d_lnP = slope;
    }
    return fma(slope, lnP - p0, k0);
  }
  // Chebyshev
  const int nT = __ldg(&r->tab_n), nP = __ldg(&r->tab_m);
  const double x = fma(__ldg(t), invT, __ldg(t + 1));
  const double y = fma(__ldg(t + 2), lnP, __ldg(t + 3));
  const double* __restrict__ a = t + 4;
  double S = 0.0, Sx = 0.0, Sy = 0.0;
  double pt0 = 1.0, pt1 = x, dt0 = 0.0, dt1 = 1.0;  // phi_t(x) and phi_t'(x)
  for (int it = 0; it < nT; it++) {
    const double pt = it == 0 ? 1.0 : pt1, dpt = it == 0 ? 0.0 : dt1;
    double B = 0.0, By = 0.0;
    double pp0 = 1.0, pp1 = y, dp0 = 0.0, dp1 = 1.0;
    for (int ip = 0; ip < nP; ip++) {
      const double pp = ip == 0 ? 1.0 : pp1, dpp = ip == 0 ? 0.0 : dp1;
      const double c = __ldg(a + it * nP + ip);
      B = fma(c, pp, B);
      if (DER) By = fma(c, dpp, By);
      if (ip >= 1) {
        const double pn = fma(2.0 * y, pp1, -pp0), dn = fma(2.0 * y, dp1, fma(2.0, pp1, -dp0));
        pp0 = pp1; pp1 = pn; dp0 = dp1; dp1 = dn;
      }
    }
    S = fma(pt, B, S);
    if (DER) {
      Sx = fma(dpt, B, Sx);
      Sy = fma(pt, By, Sy);
    }
    if (it >= 1) {
      const double pn = fma(2.0 * x, pt1, -pt0), dn = fma(2.0 * x, dt1, fma(2.0, pt1, -dt0));
      pt0 = pt1; pt1 = pn; dt0 = dt1; dt1 = dn;
    }
  }
  if (DER) {
    d_T = -Sx * __ldg(t) * invT * invT;
    d_lnP = Sy * __ldg(t + 2);
  }
  return S;
}

template <bool B>
struct BoolTag {
  static constexpr bool value = B;
};

// Temperature and pressure derivatives of ln k: d_T, d_lnP of ln k_f (the
// Arrhenius set for elementary, third-body and falloff reactions, the
// low-pressure set for chemically-activated ones, the P-log / Chebyshev forms
// otherwise) and dinf_T of ln k_inf (the Arrhenius set itself).
template <bool GEN>
__device__ __forceinline__ void ln_kf_derivatives(const DevMech& m, const Rxn* __restrict__ r, int kind, double lnT,
                                                  double invT, double invT2, double lnP, double& d_T, double& d_lnP,
                                                  double& dinf_T) {
  dinf_T = fma(__ldg(&r->theta), invT2, __ldg(&r->beta) * invT);
  d_T = dinf_T;
  d_lnP = 0.0;
  if (!GEN) return;
  if (kind >= PJ_PLOG) lnk_pdep<true>(m, r, kind, lnT, invT, lnP, d_T, d_lnP);
  else if (__ldg(&r->chem)) d_T = fma(__ldg(&r->theta0), invT2, __ldg(&r->beta0) * invT);
}

// Rate constants of one reaction: k_f, k_r (0 when irreversible) and, for
// falloff, rk = k_0 / k_inf and its log2 (2^51).
struct RateK {
  double kf, kr, rk;
  int64_t l2rk;
};

// l2rk where log2(rk) is not known in fixed point
constexpr int64_t kNoLog2 = INT64_MIN;

// The rate constants in FP64, from the stored g_k/RT (gfix: in fixed point):
// states and reactions outside the fixed point's range (A by value: its address
// taken would put it in memory).
template <bool GEN, class SA>
__device__ __noinline__ static RateK rate_constants_fp64(const DevMech& m, const SA A, int aG, const Rxn* __restrict__ r,
                                                         int kind, int rev, double lnT, double invT, double lnP,
                                                         bool gfix) {
  RateK k;
  const double lninf = fma(__ldg(&r->beta), lnT, __ldg(&r->lnA)) - __ldg(&r->theta) * invT;
  double lnkf = lninf;
  k.rk = 0.0;
  k.l2rk = kNoLog2;
  if (kind >= PJ_LINDEMANN && kind <= PJ_SRI) {
    const double ln0 = fma(__ldg(&r->beta0), lnT, __ldg(&r->lnA0)) - __ldg(&r->theta0) * invT;
    k.rk = pj_exp(ln0 - lninf);
    if (GEN && __ldg(&r->chem)) lnkf = ln0;
  }
  double u0, u1;
  if (GEN && kind >= PJ_PLOG) lnkf = lnk_pdep<false>(m, r, kind, lnT, invT, lnP, u0, u1);
  k.kf = pj_exp(lnkf);
  k.kr = 0.0;
  if (GEN && rev == 2) {
    const double* __restrict__ rt = m.tab + __ldg(&r->tab_lo);
    k.kr = pj_exp(fma(__ldg(rt + 1), lnT, __ldg(rt)) - __ldg(rt + 2) * invT);
  } else if (rev) {
    // kr = kf / Kc with Kc = exp(-sum nu g) (P_std / R T)^dnu
    const int nre = __ldg(&r->nreac), npr = __ldg(&r->nprod);
    auto g = [&](int k) {
      const double x = A.at(aG, k);
      return gfix ? fixed51_to_double(__double_as_longlong(x)) * 0.69314718055994530942 : x;
    };
    double dg = 0.0;
#pragma unroll
    for (int a = 0; a < PJ_MAX_SP; a++) {
      if (a < nre) dg = fma(-__ldg(&r->nud[a]), g(__ldg(&r->sp[a])), dg);
      if (a < npr) dg = fma(__ldg(&r->nud[PJ_MAX_SP + a]), g(__ldg(&r->sp[PJ_MAX_SP + a])), dg);
    }
    if (__ldg(&r->head.dnu_i) != 0) dg = fma(-__ldg(&r->dnu), m.log_pstd_over_r - lnT, dg);
    k.kr = pj_exp(lnkf + dg);
  }
  return k;
}

// The exponents are sums of 64-bit fixed-point terms (the sum over the
// species' Gibbs energies as integer adds), each within 2^-51 of exact, where
// FP64 terms of size 32 to 64 round at 2^-48.
template <bool GEN = true, class SA>
__device__ __forceinline__ RateK rate_constants(const DevMech& m, const SA& A, int aG, const Rxn* __restrict__ r,
                                                int kind, int rev, int nre, int npr, const FixedState& fx,
                                                double lnT, double invT, double lnP) {
  if (!fx.fast || !__ldg(&r->fx)) return rate_constants_fp64<GEN>(m, A, aG, r, kind, rev, lnT, invT, lnP, fx.fast);
  RateK k;
  int64_t y = arrhenius_fixed(__ldg(&r->head.fA), __ldg(&r->head.fB), __ldg(&r->head.fT), fx.L, fx.IT);
  k.rk = 0.0;
  k.l2rk = 0;
  if (kind >= PJ_LINDEMANN && kind <= PJ_SRI) {
    const int64_t y0 = arrhenius_fixed(__ldg(&r->fA0), __ldg(&r->fB0), __ldg(&r->fT0), fx.L, fx.IT);
    k.l2rk = y0 - y;
    k.rk = exp2_51(k.l2rk);
    if (GEN && __ldg(&r->chem)) y = y0;
  }
  k.kr = 0.0;
  if (GEN && rev == 2) {
    const double* __restrict__ rt = m.tab + __ldg(&r->tab_lo);
    k.kr = pj_exp(fma(__ldg(rt + 1), lnT, __ldg(rt)) - __ldg(rt + 2) * invT);
    rev = 0;
  }
  int64_t dg = 0;  // log2(k_r / k_f): kr = kf / Kc, Kc = exp(-sum nu g) (P_std / R T)^dnu
  if (rev) {
#pragma unroll
    for (int a = 0; a < PJ_MAX_SP; a++) {
      if (a < nre) dg -= __ldg(&r->nu[a]) * __double_as_longlong(A.at(aG, __ldg(&r->sp[a])));
      if (a < npr) dg += __ldg(&r->nu[PJ_MAX_SP + a]) * __double_as_longlong(A.at(aG, __ldg(&r->sp[PJ_MAX_SP + a])));
    }
    dg -= __ldg(&r->head.dnu_i) * fx.LP;
  }
  if (GEN && kind >= PJ_PLOG) {
    double u0, u1;
    const double lnkf = lnk_pdep<false>(m, r, kind, lnT, invT, lnP, u0, u1);
    k.kf = pj_exp(lnkf);
    if (rev) k.kr = pj_exp(fma(fixed51_to_double(dg), 0.69314718055994530942, lnkf));
    return k;
  }
  k.kf = exp2_51(y);
  if (rev) k.kr = exp2_51(y + dg);
  return k;
}

// The broadening factor of Pr = rk M and its derivatives (falloff_F); l2rk:
// log2(rk) 2^51.  MIXED: or kNoLog2, at any temperature.
template <bool DERIV, bool MIXED>
__device__ __forceinline__ void falloff_broadening(const Rxn* __restrict__ r, const LogEntry* __restrict__ log_tab,
                                                   int kind, uint64_t IT, double T, double invT, double lnT,
                                                   int64_t l2rk, double M, double Pr, double& F, double& FxPr,
                                                   double& FT) {
  F = 1.0;
  FxPr = FT = 0.0;
  if (kind == PJ_LINDEMANN) return;
  bool ok = true;
  const bool known = !MIXED || l2rk != kNoLog2;
  int64_t l2Pr = log2_51(log_tab, known ? M : Pr, ok);
  if (known) l2Pr += l2rk;
  const int fits = !MIXED || IT != 0 ? 7 : T < 65536.0 && T >= 1.0 ? 3 : 0;
  if (ok) F = falloff_F<DERIV>(log_tab, r, kind, T, invT, lnT, IT, __ldg(&r->troe_fx) & fits, l2Pr, ok, FxPr, FT);
  if (!ok) F = falloff_F_library(r, kind, T, invT, lnT, Pr, FxPr, FT);
}

// Pressure modification of a falloff reaction: Pr and, in F, FxPr, FT, the
// broadening factor and its derivatives.
template <bool DERIV>
__device__ __forceinline__ double falloff_Pr_F(const DevMech& m, const Rxn* __restrict__ r, int kind,
                                               const FixedState& fx, double T, double invT, double lnT,
                                               const RateK& k, double M, double& F, double& FxPr, double& FT) {
  const double Pr = k.rk * M;
  falloff_broadening<DERIV, true>(r, m.log_tab, kind, fx.IT, T, invT, lnT, k.l2rk, M, Pr, F, FxPr, FT);
  return Pr;
}

// Third-body concentration [M] = C_tot + sum_e (alpha_e - 1) C_e.
template <class SA>
__device__ __forceinline__ double third_body(const DevMech& m, const SA& A, int aC, const Rxn* __restrict__ r,
                                             double Ctot) {
  double M = Ctot;
  for (int e = __ldg(&r->eff_lo), eh = __ldg(&r->eff_hi); e < eh; e++) {
    if (!PJ_DBG_OK(m.dbg, e >= 0 && e < m.n_eff && __ldg(m.eff_sp + e) >= 0 && __ldg(m.eff_sp + e) < m.ns,
                   PJ_DBG_EFF))
      break;
    M = fma(__ldg(m.eff_am1 + e), A.at(aC, __ldg(m.eff_sp + e)), M);
  }
  return M;
}

__device__ __forceinline__ void red_add(double* p, double v) { atomicAdd(p, v); }  // result unused: red.global.add.f64

// wdot_k += nu_k q for the reaction's species.  k < Ns-1: nu_k L2
// reductions of +-q into wrow[k*ld] (a repeated reduction instead of a
// multiply: no FP64 instruction, which the compiler would otherwise issue,
// predicated off, for the common nu = 1 too); skipped when !w.  The bath gas,
// in few reactions (Rxn::bath_in), into a register under a branch of its own.
__device__ __forceinline__ void scatter_wdot(const Rxn* __restrict__ r, int nre, int npr, int bath, double q,
                                             double* wrow, int64_t ld, double& w_bath, bool w = true) {
  const double nq = dneg(q);
#pragma unroll
  for (int a = 0; a < PJ_MAX_SP; a++) {
    if (a < nre) {
      const int k = __ldg(&r->sp[a]);
      if (k != bath && w)
        for (int u = __ldg(&r->nu[a]); u > 0; u--) red_add(wrow + (int64_t)k * ld, nq);
    }
    if (a < npr) {
      const int k = __ldg(&r->sp[PJ_MAX_SP + a]);
      if (k != bath && w)
        for (int u = __ldg(&r->nu[PJ_MAX_SP + a]); u > 0; u--) red_add(wrow + (int64_t)k * ld, q);
    }
  }
  if (__ldg(&r->bath_in)) {
    for (int a = 0; a < PJ_MAX_SP; a++) {
      if (a < nre && __ldg(&r->sp[a]) == bath) w_bath = fma(-__ldg(&r->nud[a]), q, w_bath);
      if (a < npr && __ldg(&r->sp[PJ_MAX_SP + a]) == bath) w_bath = fma(__ldg(&r->nud[PJ_MAX_SP + a]), q, w_bath);
    }
  }
}

}  // namespace pj
