// The short path of the cooperative Jacobian kernel: one plain reaction with
// at most three factors a side, at a tile of states within the fixed point's
// range (all others: jac_reaction).
//
// What bounds it: the FP64 pipe at 16 cycles per warp instruction and SM, and
// the L2 reductions at about the same (600 G reductions/s, 15.6 cycles per
// warp instruction and SM), some 40 of which a reversible A + B = C + D
// makes.  So everything that can leave the FP64 pipe has: the exponents, the
// exponentials and the reaction enthalpy are integer fixed point, the volume
// derivative of R' = k prod C is -(number of factors) R', and an elementary
// reaction multiplies by no pressure factor: 26 FP64 instructions (23 under
// constant volume, whose S column such a reaction leaves alone) where the
// general path has 110.
#pragma once

#include "kinetics_state.cuh"
#include "source_tile.cuh"

namespace pj {

// Falloff blending c = Pr / (1 + Pr) F and its derivatives: cM = dc/dM at
// fixed T, cT = dc/dT with M moving by dMdT.  Out of line, as falloff_factor.
struct FalloffC {
  double c, cM, cT;
};
template <bool MIXED>
__device__ __noinline__ static FalloffC falloff_derivatives(const Rxn* __restrict__ r,
                                                            const LogEntry* __restrict__ log_tab, int kind, double T,
                                                            double invT, double lnT, uint64_t IT, double rk,
                                                            int64_t l2rk, double M, double dMdT) {
  double F, FxPr, FT;
  const double Pr = rk * M;
  falloff_broadening<true, MIXED>(r, log_tab, kind, IT, T, invT, lnT, l2rk, M, Pr, F, FxPr, FT);
  const double invT2 = invT * invT;
  const double dlnrk = fma(__ldg(&r->theta0) - __ldg(&r->theta), invT2, (__ldg(&r->beta0) - __ldg(&r->beta)) * invT);
  const double i1p = inverse_1p(Pr);
  const double fr = Pr * i1p;
  const double cPr = F * i1p * i1p + FxPr * i1p;
  return FalloffC{fr * F, cPr * rk, fr * FT + cPr * (Pr * dlnrk + rk * dMdT)};
}

// sum nu h/RT - d over a short-path reaction's factors; H: this lane's h_k/RT
// (enthalpy_entry), 32 words per species
template <bool MIXED>
__device__ __forceinline__ double lean_energy(const RxnHead& h, const double* __restrict__ H, int d, bool fast) {
  if (MIXED && !fast) return lean_sum(h, H, (double)d);
  auto hf = [&](int off) { return __double_as_longlong(H[off]); };
  int64_t s = hf(h.b[0]) - hf(h.f[0]) - ((int64_t)d << 51);
  if (h.nf > 1) s -= hf(h.f[1]);
  if (h.nb > 1) s += hf(h.b[1]);
  if (h.nf > 2) s -= hf(h.f[2]);
  if (h.nb > 2) s += hf(h.b[2]);
  return fixed51_to_double(s);
}

// x in the derivative type.  To FP32 in integer instructions (the hardware
// conversion takes an FP64-pipe slot): rounded to nearest, flushed to zero
// below 2^-126, infinite beyond FP32's range, NaN for NaN.
template <typename DT>
__device__ __forceinline__ DT to_derivative(double x) {
  if constexpr (sizeof(DT) == 8) {
    return x;
  } else {
    const uint64_t b = (uint64_t)__double_as_longlong(x) + 0x10000000ull;
    const int e = (int)((uint32_t)(b >> 52) & 0x7ffu) - 896;
    uint32_t f = ((uint32_t)e << 23) | ((uint32_t)(b >> 29) & 0x7fffffu);
    f = e < 1 ? 0u : f;
    f = e > 254 ? 0x7f800000u : f;
    if (e == 1151) f |= (uint32_t)(b >> 29) & 0x7fffffu;  // infinity, or NaN (quiet: a high fraction bit is set)
    return __uint_as_float(f | ((uint32_t)__double2hiint(x) & 0x80000000u));
  }
}

__device__ __forceinline__ int shape_species(int shape) { return shape <= SH_2 ? 1 : shape <= SH_21 ? 2 : 3; }

// x with its sign bit flipped by a mask (0 or 0x80000000)
__device__ __forceinline__ double flip(double x, uint32_t sign) {
  return __hiloint2double((int)((uint32_t)__double2hiint(x) ^ sign), __double2loint(x));
}
__device__ __forceinline__ float flip(float x, uint32_t sign) { return __uint_as_float(__float_as_uint(x) ^ sign); }

// base: this lane's column of the tile's arrays C, g, h ([3][ns][32]).
template <int MODE, int FMT, typename DT, bool NEWTON>
__device__ __forceinline__ void lean_jacobian(const DevMech& m, const Rxn* __restrict__ r, const RxnHead& h,
                                              const double* __restrict__ base, JacVars<DT>& v, const JacOut<DT>& o) {
  const int ns = m.ns, bath = ns - 1;
  const double* __restrict__ C = base;
  const double* __restrict__ G = base + ns * kTile;
  const double* __restrict__ H = base + 2 * ns * kTile;
  RxnJac a;
  {
    const int4* __restrict__ p = reinterpret_cast<const int4*>(&r->jac);
    int4* q = reinterpret_cast<int4*>(&a);
#pragma unroll
    for (int i = 0; i < 4; i++) q[i] = __ldg(p + i);
  }
  const bool rev = h.rev != 0;
  const LeanK k = lean_constants<false>(m, r, h, G, v.fx, v.lnT, v.invT);
  // both sides, the net rate and V dRn/dV at constant n, -(factors) R by side
  LeanSide sf, sb;
  double Rn, VS;
  lean_shapes(h.code, [&](auto tf, auto tb) {
    constexpr int SF = decltype(tf)::value, SB = decltype(tb)::value;
    constexpr int nfac[5] = {1, 2, 2, 3, 3};
    sf = lean_side<SF>(h.f, C, k.kf);
    sb = lean_side<SB>(h.b, C, k.kr);
    Rn = SB < 0 ? sf.R : sf.R - sb.R;
    VS = 0.0;
    if (MODE == PJ_CONP) {
      constexpr int NF = nfac[SF], NB = SB < 0 ? NF : nfac[SB < 0 ? 0 : SB];
      if (NF == NB) VS = NF == 1 ? dneg(Rn) : -(double)NF * Rn;
      else VS = (NB == 1 ? sb.R : (double)NB * sb.R) - (NF == 1 ? sf.R : (double)NF * sf.R);
    }
  });

  const double de = lean_energy<false>(h, H, h.dnu_i, true);  // sum nu h/RT - dnu
  double dhd = de;
  if (MODE == PJ_CONP && h.dnu_i != 0) dhd = lean_energy<false>(h, H, 0, true);

  // T derivative of the net rate: T d ln kf/dT = Ef = beta + theta/T, T d ln
  // kr/dT = Ef - de, so T dRn/dT = Rn Ef + Rr de; times V
  const double Ef = fma(a.theta, v.invT, a.beta);
  double VT = fma(sb.R, de, Rn * Ef) * (v.V * v.invT);
  double Gb = 0.0;  // dRn/dC of the bath gas itself
  bool has_S = MODE == PJ_CONP;
  if (a.bath) {
    if (a.bath & 1) Gb += sf.d0;
    if (a.bath & 2) Gb += sf.d1;
    if (a.bath & 4) Gb += sf.d2;
    if (a.bath & 8) Gb -= sb.d0;
    if (a.bath & 16) Gb -= sb.d1;
    if (a.bath & 32) Gb -= sb.d2;
    VT = fma(Gb, v.V * v.dCb_T, VT);
    if (MODE == PJ_CONP) VS = a.nbx * sb.R - a.nfx * sf.R;  // the bath gas's concentration is not n/V
    VS = fma(Gb, v.V * v.dCb_S, VS);
    has_S = true;
  }

  // pressure factor: scales the rate and every derivative
  double q = Rn;
  double RcM = 0.0;  // Rn dc/dM
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
    double cT = dMdT, c = M;
    RcM = Rn;
    if (h.kind != PJ_THIRD_BODY) {
      int64_t l2rk;
      const double rk = lean_falloff<false>(r, k, v.fx, v.lnT, v.invT, l2rk);
      const FalloffC fc =
          falloff_derivatives<false>(r, m.log_tab, h.kind, v.T, v.invT, v.lnT, v.fx.IT, rk, l2rk, M, dMdT);
      c = fc.c;
      cT = fc.cT;
      RcM = Rn * fc.cM;
    }
    q = c * Rn;
    VT = fma(c, VT, (Rn * cT) * v.V);
    VS = fma(c, VS, (RcM * dMdS) * v.V);
    has_S = true;
    Gb *= c;
    sf.d0 *= c;
    sf.d1 *= c;
    sf.d2 *= c;
    sb.d0 *= c;
    sb.d1 *= c;
    sb.d2 *= c;
  }

  // energy- and state-row weights of this reaction
  const DT dE = to_derivative<DT>((RU * v.T) * (MODE == PJ_CONP ? dhd : de));
  const DT dW = DT(a.dW);
  const DT VT_t = to_derivative<DT>(VT);
  v.AT_T = v.AT_T + dE * VT_t;
  v.AS_T = v.AS_T + dW * VT_t;
  const DT jT = nscale<NEWTON>(o, VT_t);
  DT jS = DT(0);
  if (has_S) {
    const DT VS_t = to_derivative<DT>(VS);
    v.AT_S = v.AT_S + dE * VS_t;
    v.AS_S = v.AS_S + dW * VS_t;
    jS = nscale<NEWTON>(o, VS_t);
  }

  // Jacobian entries and production rates, by L2 reductions.  Addresses: an
  // entry's row of ld values, 32 x 32 -> 64 bit (the caller checks that ld
  // fits); up to four rows unrolled with their signs as masks.
  DT B_t = DT(0);
  if (o.w) {
    const int32_t* __restrict__ tg = (FMT == PJ_CSR ? m.tgt_csr : m.tgt_csc) + a.tgt_lo;
    const RowNu* __restrict__ rows = m.rows + a.row_lo;
    const int nrows = a.nrows;
    const uint32_t ldJ = (uint32_t)o.ld * (uint32_t)sizeof(DT), ldw = (uint32_t)o.ld * 8u;
    char* const Jb = reinterpret_cast<char*>(o.J + o.s);
    char* const wb = reinterpret_cast<char*>(o.wrow);
    uint32_t sg[4];
#pragma unroll
    for (int p = 0; p < 4; p++) sg[p] = (uint32_t)a.neg << (31 - p) & 0x80000000u;
    auto red = [&](int e, DT x) {
      if (!PJ_DBG_OK(m.dbg, e >= 0 && e < (FMT == PJ_DENSE ? m.N * m.N : m.nnz), PJ_DBG_TARGET)) return;
      red_add(reinterpret_cast<DT*>(Jb + (uint64_t)(uint32_t)e * ldJ), x);
    };
    auto row = [&](int p, int k, uint32_t sign) {
      red(FMT == PJ_DENSE ? (k + 2) * m.N : __ldg(tg + 2 * p), flip(jT, sign));
      if (has_S) red(FMT == PJ_DENSE ? (k + 2) * m.N + 1 : __ldg(tg + 2 * p + 1), flip(jS, sign));
      red_add(reinterpret_cast<double*>(wb + (uint64_t)(uint32_t)k * ldw), flip(q, sign));
    };
#pragma unroll
    for (int p = 0; p < 4; p++)
      if (p < nrows) row(p, a.k[p], sg[p]);
    for (int p = 4; p < nrows; p++) row(p, __ldg(&rows[p].k), (uint32_t)a.neg << (31 - p) & 0x80000000u);
    tg += 2 * nrows;

    // species columns
    auto slot = [&](int j, DT val) {
      const DT vs = nscale<NEWTON>(o, val);
      red(FMT == PJ_DENSE ? j + 2 : __ldg(tg), dE * vs);
      red(FMT == PJ_DENSE ? m.N + j + 2 : __ldg(tg + 1), dW * vs);
#pragma unroll
      for (int p = 0; p < 4; p++)
        if (p < nrows) red(FMT == PJ_DENSE ? (a.k[p] + 2) * m.N + j + 2 : __ldg(tg + 2 + p), flip(vs, sg[p]));
      for (int p = 4; p < nrows; p++)
        red(FMT == PJ_DENSE ? (__ldg(&rows[p].k) + 2) * m.N + j + 2 : __ldg(tg + 2 + p),
            flip(vs, (uint32_t)a.neg << (31 - p) & 0x80000000u));
      tg += nrows + 2;
    };
    const int nsf = shape_species(a.shape[0]), nsb = rev ? shape_species(a.shape[1]) : 0;
#pragma unroll
    for (int s = 0; s < 3; s++) {
      if (s < nsf && !(a.bath >> s & 1))
        slot(FMT == PJ_DENSE ? __ldg(&r->sp[s]) : 0, to_derivative<DT>(s == 0 ? sf.d0 : s == 1 ? sf.d1 : sf.d2));
      if (s < nsb && !(a.bath >> (3 + s) & 1))
        slot(FMT == PJ_DENSE ? __ldg(&r->sp[PJ_MAX_SP + s]) : 0,
             dneg(to_derivative<DT>(s == 0 ? sb.d0 : s == 1 ? sb.d1 : sb.d2)));
    }
    double Bi = -Gb;  // minus the terms of the bath gas
    if (h.kind != PJ_ELEMENTARY) {
      for (int e = __ldg(&r->eff_lo), eh = __ldg(&r->eff_hi); e < eh; e++) {
        if (!PJ_DBG_OK(m.dbg, e >= 0 && e < m.n_eff, PJ_DBG_EFF)) break;
        const int j = __ldg(m.eff_sp + e);
        const double val = RcM * __ldg(m.eff_am1 + e);
        if (j == bath) Bi -= val;
        else slot(j, to_derivative<DT>(val));
      }
    }
    if (a.dense) {
      B_t = to_derivative<DT>(Bi);
      const DT Bs = nscale<NEWTON>(o, B_t);
      for (int p = 0; p < nrows; p++) {
        const int k = __ldg(&rows[p].k);
        const DT val = flip(Bs, (uint32_t)a.neg << (31 - p) & 0x80000000u);
        if (FMT == PJ_CSR) {
          // a dense row holds every species column, contiguous in CSR
          const int64_t e2 = jpos<FMT>(m, k + 2, 2);
          if (!PJ_DBG_OK(m.dbg, e2 >= 0 && e2 + ns - 1 <= m.nnz, PJ_DBG_POSMAP)) continue;
          for (int j = 0; j < ns - 1; j++) red((int)e2 + j, val);
        } else {
          for (int j = 0; j < ns - 1; j++) red((int)jpos<FMT>(m, k + 2, j + 2), val);
        }
      }
    }
  }
  if (a.dense) {
    v.ATB = v.ATB + dE * B_t;
    v.ASB = v.ASB + dW * B_t;
  }
  if (a.bath) {  // the bath gas's own production rate: net coefficient times q
    int nu = 0;
#pragma unroll
    for (int s = 0; s < 3; s++) {
      if (s < h.nf && h.f[s] == kTile * bath) nu--;
      if (s < h.nb && h.b[s] == kTile * bath) nu++;
    }
    v.w_bath = fma((double)nu, q, v.w_bath);
  }
}

}  // namespace pj
