// Source terms of a tile of 32 states by the warps of one block (lane =
// state): the shared body of the source-term, eval_y and finite-difference
// kernels.
//
// What bounds it: the FP64 pipe (16 cycles per warp instruction and SM) and
// the integer pipes that evaluate the exponentials.  The tile's C_k and
// g_k/RT sit once in shared memory (a warp's access to one species is 32
// consecutive 8-byte words), so 16 warps work on one state set that one warp
// per state set would spill to L2, and a small batch uses 16 warps per 32
// states.
//
// Deterministic: reaction i's net rate q_i goes to a shared buffer (a chunk
// of kGatherChunk reactions, double-buffered), and the warp that owns species
// k adds the chunk's contributions to k's production rate in kernel order,
// as L2 reductions into an accumulator row (the additions run at L2, not on
// the SM's FP64 pipe; one thread's reductions to one address apply in its
// program order).  Every cross-warp sum is a sum of per-warp partials in
// warp order.  The result does not depend on the launch shape.
#pragma once

#include "kinetics_common.cuh"

namespace pj {

constexpr int kTile = 32;
constexpr int kSrcWarps = 16;  // warps per block, or twice that

enum SrcSc { zT, zV, zP, zInvT, zInvV, zLnT, zLnP, zCtot, zL, zIT, zLP, zCdum, zDen, zCxB, kSrcSc };
enum SrcPart { rAcc, rDen, rNum, rOm, kSrcPart };
enum SrcFlag { gOk, gFast, kSrcFlag };  // gFast: 1 in the fixed point's range; 0: T out of it; 2: some g_k

__host__ __device__ constexpr size_t source_arrays_bytes(int ns) { return (size_t)2 * ns * kTile * sizeof(double); }
__host__ __device__ constexpr size_t source_smem_bytes(int ns, bool arrays_smem) {
  return (arrays_smem ? source_arrays_bytes(ns) : 0) +
         (size_t)(2 * kGatherChunk + kSrcSc + kSrcPart * kSrcWarps) * kTile * sizeof(double) +
         (size_t)kSrcFlag * kTile * sizeof(int);
}
// C_k and g_k/RT in a global workspace where they do not fit in shared memory
__host__ __device__ constexpr size_t source_arrays_ws_doubles(int ns, bool arrays_smem) {
  return arrays_smem ? 0 : (size_t)2 * ns * kTile;
}

// Pressure factor of a reaction with a third body: [M], or the falloff
// blending (Pr / (1 + Pr)) F; chem: chemically activated, F / (1 + Pr).  Out
// of line: it runs for about a fifth of the reactions, and its registers
// would otherwise set every reaction's.
template <bool MIXED>
__device__ __noinline__ static double falloff_factor(const Rxn* __restrict__ r, const LogEntry* __restrict__ log_tab,
                                                     int kind, double T, double invT, double lnT, uint64_t IT, double rk,
                                                     int64_t l2rk, double M, bool chem) {
  double F, d1, d2;
  const double Pr = rk * M;
  falloff_broadening<false, MIXED>(r, log_tab, kind, IT, T, invT, lnT, l2rk, M, Pr, F, d1, d2);
  const double i1p = inverse_1p(Pr);
  return (chem ? i1p : Pr * i1p) * F;
}

// The warp-uniform head of a reaction's record.
__device__ __forceinline__ RxnHead load_head(const Rxn* __restrict__ r) {
  RxnHead h;
  const int4* __restrict__ p = reinterpret_cast<const int4*>(&r->head);
  int4* q = reinterpret_cast<int4*>(&h);
#pragma unroll
  for (int i = 0; i < 4; i++) q[i] = __ldg(p + i);
  return h;
}

// log2(k_r / k_f) 2^51 of a short-path reversible reaction; G: this lane's
// g_k/RT (gibbs_entry, in range), 32 words per species.
__device__ __forceinline__ int64_t lean_gibbs(const RxnHead& h, const double* __restrict__ G, int64_t LP) {
  auto g = [&](int off) { return __double_as_longlong(G[off]); };
  int64_t s = g(h.b[0]) - g(h.f[0]);
  if (h.nf > 1) s -= g(h.f[1]);
  if (h.nb > 1) s += g(h.b[1]);
  if (h.nf > 2) s -= g(h.f[2]);
  if (h.nb > 2) s += g(h.b[2]);
  if (h.dnu_i != 0) s -= (int64_t)h.dnu_i * LP;
  return s;
}

// sum nu x over a short-path reaction's factors, less d, of FP64 entries
__device__ __forceinline__ double lean_sum(const RxnHead& h, const double* __restrict__ x, double d) {
  double s = x[h.b[0]] - x[h.f[0]] - d;
  if (h.nf > 1) s -= x[h.f[1]];
  if (h.nb > 1) s += x[h.b[1]];
  if (h.nf > 2) s -= x[h.f[2]];
  if (h.nb > 2) s += x[h.b[2]];
  return s;
}

// Rate constants of a short-path reaction.  MIXED: in a tile where some state
// is outside the fixed point's range, each lane by its own state, the others
// in FP64; what follows them is the same code for every lane, so that a
// state's result does not depend on its tile mates.
struct LeanK {
  double kf, kr;
  int64_t y;  // log2(kf) 2^51; kNoLog2 in FP64
};
template <bool MIXED>
__device__ __forceinline__ LeanK lean_constants(const DevMech& m, const Rxn* __restrict__ r, const RxnHead& h,
                                                const double* __restrict__ G, const FixedState& fx, double lnT,
                                                double invT) {
  LeanK k;
  k.kr = 0.0;
  if (!MIXED || fx.fast) {
    k.y = arrhenius_fixed(h.fA, h.fB, h.fT, fx.L, fx.IT);
    k.kf = exp2_51(k.y);
    if (h.rev) k.kr = exp2_51(k.y + lean_gibbs(h, G, fx.LP));
  } else {
    k.y = kNoLog2;
    const double lnkf = fma(__ldg(&r->beta), lnT, __ldg(&r->lnA)) - __ldg(&r->theta) * invT;
    k.kf = pj_exp(lnkf);
    if (h.rev) {
      double dg = lean_sum(h, G, 0.0);
      if (h.dnu_i != 0) dg = fma(-__ldg(&r->dnu), m.log_pstd_over_r - lnT, dg);
      k.kr = pj_exp(lnkf + dg);
    }
  }
  return k;
}

// rk = k_0 / k_inf of a short-path falloff reaction and its log2 2^51 (or
// kNoLog2), from its k_inf.
template <bool MIXED>
__device__ __forceinline__ double lean_falloff(const Rxn* __restrict__ r, const LeanK& k, const FixedState& fx,
                                               double lnT, double invT, int64_t& l2rk) {
  if (!MIXED || fx.fast) {
    l2rk = arrhenius_fixed(__ldg(&r->fA0), __ldg(&r->fB0), __ldg(&r->fT0), fx.L, fx.IT) - k.y;
    return exp2_51(l2rk);
  }
  l2rk = kNoLog2;
  return pj_exp((fma(__ldg(&r->beta0), lnT, __ldg(&r->lnA0)) - __ldg(&r->theta0) * invT) -
                (fma(__ldg(&r->beta), lnT, __ldg(&r->lnA)) - __ldg(&r->theta) * invT));
}

// One side's product R = k prod C and dR/dC_a in species order (f: factors
// as packed in the head; unused derivatives are left 0).
struct LeanSide {
  double R, d0, d1, d2;
};
template <int SHAPE>
__device__ __forceinline__ LeanSide lean_side(const int32_t (&f)[3], const double* __restrict__ C, double k) {
  LeanSide s{0.0, 0.0, 0.0, 0.0};
  if constexpr (SHAPE < 0) return s;
  const double c0 = C[f[0]];
  if constexpr (SHAPE == SH_1) {
    s.R = k * c0;
    s.d0 = k;
  } else if constexpr (SHAPE == SH_11 || SHAPE == SH_2) {
    const double t = k * c0, c1 = C[f[1]];
    s.R = t * c1;
    s.d0 = SHAPE == SH_2 ? t + t : t;
    if (SHAPE == SH_11) s.d1 = k * c1;
  } else if constexpr (SHAPE >= 0) {
    const double t = k * c0, c1 = C[f[1]], c2 = C[f[2]];
    const double t1 = t * c1;
    s.R = t1 * c2;
    s.d0 = SHAPE == SH_21 ? t1 + t1 : t1;  // 2A + B as A B A, A + B + C as C B A
    s.d1 = t * c2;
    if (SHAPE == SH_111) s.d2 = (k * c2) * c1;
  }
  return s;
}

// f(forward shape, reverse shape or -1) with the shapes of a head's code as
// compile-time constants.  A jump table: under conditions of its own each
// shape's few FP64 instructions would be predicated, and the FP64 pipe
// charges a predicated-off warp instruction like any other (20 of the 63 a
// 53-species Jacobian reaction issued).  Short-path reactions only: pack_head
// gives no other the flag, and theirs no code beyond the table.
template <int V>
struct IntTag {
  static constexpr int value = V;
};
template <class F>
__device__ __forceinline__ void lean_shapes(int code, F&& f) {
  switch (code) {
#define PJ_SHAPE(sf, sb) \
  case 6 * (sf) + 1 + (sb): f(IntTag<sf>{}, IntTag<sb>{}); break;
#define PJ_SHAPES(sf) PJ_SHAPE(sf, -1) PJ_SHAPE(sf, 0) PJ_SHAPE(sf, 1) PJ_SHAPE(sf, 2) PJ_SHAPE(sf, 3) PJ_SHAPE(sf, 4)
    PJ_SHAPES(0)
    PJ_SHAPES(1)
    PJ_SHAPES(2)
    PJ_SHAPES(3)
    PJ_SHAPES(4)
#undef PJ_SHAPES
#undef PJ_SHAPE
    default: break;
  }
}

// Net rate of reaction i at this lane's state, short path: a plain reaction
// with at most three factors a side.
template <bool MIXED>
__device__ __forceinline__ double lean_rate(const DevMech& m, const Rxn* __restrict__ r, const RxnHead& h,
                                            const double* __restrict__ C, const double* __restrict__ G,
                                            const FixedState& fx, double T, double invT, double lnT, double Ctot) {
  const LeanK k = lean_constants<MIXED>(m, r, h, G, fx, lnT, invT);
  double q = 0.0;
  lean_shapes(h.code, [&](auto sf, auto sb) {
    q = lean_side<decltype(sf)::value>(h.f, C, k.kf).R;
    if (decltype(sb)::value >= 0) q -= lean_side<decltype(sb)::value>(h.b, C, k.kr).R;
  });
  if (h.kind != PJ_ELEMENTARY) {
    double M = Ctot;
    for (int e = __ldg(&r->eff_lo), eh = __ldg(&r->eff_hi); e < eh; e++) {
      if (!PJ_DBG_OK(m.dbg, e >= 0 && e < m.n_eff && __ldg(m.eff_sp + e) >= 0 && __ldg(m.eff_sp + e) < m.ns,
                     PJ_DBG_EFF))
        break;
      M = fma(__ldg(m.eff_am1 + e), C[kTile * __ldg(m.eff_sp + e)], M);
    }
    if (h.kind == PJ_THIRD_BODY) {
      q *= M;
    } else {
      int64_t l2rk;
      const double rk = lean_falloff<MIXED>(r, k, fx, lnT, invT, l2rk);
      q *= falloff_factor<MIXED>(r, m.log_tab, h.kind, T, invT, lnT, fx.IT, rk, l2rk, M, false);
    }
  }
  return q;
}

// What the reactions read of the state besides C and g (sc: this lane's scalars
// of the tile).
struct SrcVars {
  FixedState fx;
  double T, invT, lnT, lnP, Ctot;
};
__device__ __forceinline__ SrcVars source_vars(const double* __restrict__ sc, bool fast) {
  auto S = [&](int v) { return sc[v * kTile]; };
  SrcVars v;
  v.T = S(zT);
  v.invT = S(zInvT);
  v.lnT = S(zLnT);
  v.lnP = S(zLnP);
  v.Ctot = S(zCtot);
  v.fx.L = (uint64_t)__double_as_longlong(S(zL));
  v.fx.IT = (uint64_t)__double_as_longlong(S(zIT));
  v.fx.LP = __double_as_longlong(S(zLP));
  v.fx.fast = fast;
  return v;
}

// Net rate of any reaction at any state.  Out of line (special types, sides
// of more than three factors).
template <bool SPECIAL>
__device__ __noinline__ static double general_rate(const DevMech& m, double* base, const double* sc,
                                                   const Rxn* __restrict__ r, bool fast) {
  const SrcVars v = source_vars(sc, fast);
  const FixedState& fx = v.fx;
  const double T = v.T, invT = v.invT, lnT = v.lnT, lnP = v.lnP, Ctot = v.Ctot;
  StateArrays A;
  A.ns = m.ns;
  A.base = base;
  A.stride = kTile;
  enum { aC = 0, aG = 1 };
  const int kind = __ldg(&r->kind);
  const int nre = __ldg(&r->nreac), npr = __ldg(&r->nprod), rev = __ldg(&r->rev);
  const RateK k = rate_constants<SPECIAL>(m, A, aG, r, kind, rev, nre, npr, fx, lnT, invT, lnP);
  double dmy[PJ_MAX_SP];
  const double Rf = side_rate<false>(A, aC, r, 0, __ldg(&r->shape[0]), nre, k.kf, dmy);
  const double Rr = rev ? side_rate<false>(A, aC, r, PJ_MAX_SP, __ldg(&r->shape[1]), npr, k.kr, dmy) : 0.0;
  double c = 1.0;
  if (has_third_body(kind)) {
    const double M = third_body(m, A, aC, r, Ctot);
    c = kind == PJ_THIRD_BODY
            ? M
            : falloff_factor<true>(r, m.log_tab, kind, T, invT, lnT, fx.IT, k.rk, k.l2rk, M, SPECIAL && __ldg(&r->chem));
  }
  return c * (Rf - Rr);
}

// Net rates of a warp's reactions first, first + step, .. < end, into q, in a
// tile with a state outside the fixed point's range.  The whole loop out of
// line and the state read again from shared memory, so that the short path
// beside it is compiled as if it were alone (53 species, 1 Mi states: 11.58 ms
// with and without it).
template <bool SPECIAL>
__device__ __noinline__ static void mixed_rates(const DevMech& m, double* base, const double* sc, double* q, bool fast,
                                                int first, int step, int end) {
  const SrcVars v = source_vars(sc, fast);
  for (int i = first; i < end; i += step, q += step * kTile) {
    const Rxn* __restrict__ r = m.rxn + i;
    const RxnHead h = load_head(r);
    *q = h.lean ? lean_rate<true>(m, r, h, base, base + m.ns * kTile, v.fx, v.T, v.invT, v.lnT, v.Ctot)
                : general_rate<SPECIAL>(m, base, sc, r, fast);
  }
}

// One tile.  In: act() (this lane has a state), T(), S(), par(), n(k); Out:
// acc(k) (this lane's production-rate accumulator of species k, not touched
// where !act()), species(k, V, wk) for every k (the bath gas too), head(Tdot,
// Sdot), invalid().  smem: source_smem_bytes; arrays: this block's
// source_arrays_ws_doubles, or null with the arrays in shared memory; AS: kShared
// or kGlobal where that is known at compile time (shared-memory addressing in
// place of generic loads), else kEither.  Every thread of the block calls it.
enum ArraySpace { kShared, kGlobal, kEither };
template <int MODE, bool SPECIAL, int AS, class In, class Out>
__device__ __forceinline__ void source_tile(const DevMech& m, double* smem, double* arrays, const In& in,
                                            const Out& out) {
  const int ns = m.ns, bath = m.ns - 1, nr = m.nr;
  const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  // species are split over the first 16 warps whatever the block's size, so
  // that the result does not depend on it
  constexpr int W = kSrcWarps;
  const int W_all = blockDim.x >> 5;
  double* const base = (AS == kShared ? smem : AS == kGlobal ? arrays : arrays ? arrays : smem) + lane;  // C then g, [2][ns][32]
  double* const C = base;
  double* const G = base + ns * kTile;
  double* const qbuf = smem + (AS == kGlobal || (AS == kEither && arrays) ? 0 : 2 * ns * kTile) + lane;
  double* const sc = qbuf + 2 * kGatherChunk * kTile;
  double* const part = sc + kSrcSc * kTile;
  int* const flags = reinterpret_cast<int*>(part - lane + kSrcPart * W * kTile) + lane;
  auto S = [&](int v) -> double& { return sc[v * kTile]; };
  auto Pw = [&](int w, int v) -> double& { return part[(w * kSrcPart + v) * kTile]; };
  auto sum_parts = [&](int v) {
    double t = 0.0;
    for (int w = 0; w < W; w++) t += Pw(w, v);
    return t;
  };
  const bool act = in.act();

  // A: the state's scalars (warp 0; a lane without a valid T, V, P takes a
  // dummy state); zero accumulators
  if (warp == 0) {
    double T = 1000.0, V = 1.0, P = 1e5;
    bool ok0 = false;
    if (act) {
      const double T_ = in.T(), S_ = in.S(), par = in.par();
      const double V_ = MODE == PJ_CONP ? S_ : par, P_ = MODE == PJ_CONP ? par : S_;
      ok0 = (T_ > 0.0) && (V_ > 0.0) && (P_ > 0.0) && isfinite(T_) && isfinite(V_) && isfinite(P_);
      if (ok0) {
        T = T_;
        V = V_;
        P = P_;
      }
    }
    const double invT = 1.0 / T;
    double lnT;
    FixedState fx;
    temperature_terms(m, T, invT, lnT, fx);
    const double Ctot = P / (RU * T);
    S(zT) = T;
    S(zV) = V;
    S(zP) = P;
    S(zInvT) = invT;
    S(zInvV) = 1.0 / V;
    S(zLnT) = lnT;
    S(zLnP) = m.has_pdep ? log(P) : 0.0;
    S(zCtot) = Ctot;
    S(zL) = __longlong_as_double((long long)fx.L);
    S(zIT) = __longlong_as_double((long long)fx.IT);
    S(zLP) = __longlong_as_double((long long)fx.LP);
    S(zCdum) = Ctot / ns;
    flags[gOk * kTile] = ok0;
    flags[gFast * kTile] = fx.fast;
  }
  if (act && warp < W)
    for (int k = warp; k < ns; k += W) *out.acc(k) = 0.0;
  __syncthreads();

  // B: concentrations and thermo of the warp's species
  if (warp < W) {
    const double T = S(zT), invT = S(zInvT), lnT = S(zLnT), cdum = S(zCdum), V = S(zV), invV = S(zInvV);
    const bool ok0 = flags[gOk * kTile] != 0;
    double acc = 0.0, den = 0.0;
    const bool fast0 = flags[gFast * kTile] != 0;
    bool fast = fast0;
    for (int k = warp; k < ns; k += W) {
      double cp, g;
      nasa_cp_g(nasa_block(m, k, T), T, invT, lnT, cp, g);
      G[k * kTile] = gibbs_entry(m, g, fast);
      const double cx = MODE == PJ_CONP ? cp : cp - 1.0;
      if (k < bath) {
        const double c = ok0 ? concentration(in.n(k), V, invV) : cdum;
        C[k * kTile] = c;
        acc += c;
        den = fma(c, cx, den);
      } else {
        S(zCxB) = cx;
      }
    }
    if (fast0 && !fast) flags[gFast * kTile] = 2;  // found out of range part of the way
    Pw(warp, rAcc) = acc;
    Pw(warp, rDen) = den;
  }
  __syncthreads();

  // C: bath gas by subtraction, validity, the energy equation's denominator;
  // the entries of a state found out of range, again
  if (warp < W && flags[gFast * kTile] == 2) {
    const double T = S(zT), invT = S(zInvT), lnT = S(zLnT);
    for (int k = warp; k < ns; k += W) {
      double cp, g;
      nasa_cp_g(nasa_block(m, k, T), T, invT, lnT, cp, g);
      G[k * kTile] = g;
    }
  }
  if (warp == 0) {
    const double Ctot = S(zCtot);
    const double acc = sum_parts(rAcc);
    const double Cns = Ctot - acc;
    const bool ok = flags[gOk * kTile] != 0 && isfinite(acc) && isfinite(Cns) && !(Cns < -1e-12 * Ctot);
    C[bath * kTile] = Cns;
    S(zDen) = RU * (sum_parts(rDen) + Cns * S(zCxB));
    flags[gOk * kTile] = ok;
  }
  __syncthreads();

  // D: the reactions, by chunks; then the chunk's contributions to the
  // warp's species
  {
    const bool fast = flags[gFast * kTile] == 1;
    const SrcVars v = source_vars(sc, fast);
    const bool fast_tile = __all_sync(0xffffffffu, fast);  // the same in every warp
    int chunk = 0;
    for (int c0 = 0; c0 < nr; c0 += kGatherChunk, chunk++) {
      double* const q = qbuf + (chunk & 1) * kGatherChunk * kTile;
      const int c1 = min(nr, c0 + kGatherChunk);
      if (fast_tile) {
        for (int i = c0 + warp; i < c1; i += W_all) {
          const Rxn* __restrict__ r = m.rxn + i;
          const RxnHead h = load_head(r);
          q[(i - c0) * kTile] = h.lean ? lean_rate<false>(m, r, h, C, G, v.fx, v.T, v.invT, v.lnT, v.Ctot)
                                       : general_rate<SPECIAL>(m, base, sc, r, fast);
        }
      } else {
        mixed_rates<SPECIAL>(m, base, sc, q + warp * kTile, fast, c0 + warp, W_all, c1);
      }
      __syncthreads();
      for (int k = warp; k < ns; k += W_all) {
        const int32_t* __restrict__ gp = m.gather_ptr + (size_t)chunk * ns + k;
        for (int e = __ldg(gp), e1 = __ldg(gp + 1); e < e1; e++) {
          const uint32_t id = __ldg(m.gather + e);
          if (!PJ_DBG_OK(m.dbg, (int)(id & 0x7fffu) < c1 - c0, PJ_DBG_ROWS)) break;
          const double v = q[(id & 0x7fffu) * kTile];
          if (act) red_add(out.acc(k), id & 0x8000u ? dneg(v) : v);
        }
      }
    }
  }

  // E: the warp's species (with 16 warps, their accumulators only this warp
  // has touched)
  if (W_all > W) __syncthreads();
  if (warp < W) {
    const double T = S(zT), invT = S(zInvT), V = S(zV);
    const bool ok = flags[gOk * kTile] != 0;
    double num = 0.0, Om = 0.0;
    for (int k = warp; k < ns; k += W) {
      const double h = nasa_h(nasa_block(m, k, T), T, invT);
      const double wk = act ? __ldcg(out.acc(k)) : 0.0;
      num = fma(MODE == PJ_CONP ? h : h - 1.0, wk, num);
      if (k < bath) Om = fma(__ldg(m.wfac + k), wk, Om);
      if (act && ok) out.species(k, V, wk);
    }
    Pw(warp, rNum) = num;
    Pw(warp, rOm) = Om;
  }
  __syncthreads();

  // F: the energy equation and the ideal-gas state equation (warp 0)
  if (warp == 0) {
    const double T = S(zT), invT = S(zInvT), V = S(zV), P = S(zP);
    const double num = sum_parts(rNum) * (RU * T), Om = sum_parts(rOm);
    const double Tdot = -num / S(zDen);
    const double Sdot = MODE == PJ_CONP ? V * Tdot * invT + (RU * T * V / P) * Om : P * Tdot * invT + RU * T * Om;
    if (act) {
      if (flags[gOk * kTile]) out.head(Tdot, Sdot);
      else out.invalid();
    }
  }
}

// States of one batch: lane s of the tile.
struct BatchIn {
  const double* __restrict__ param;
  const double* __restrict__ phi;
  int64_t ld, s;
  bool active;
  __device__ __forceinline__ bool act() const { return active; }
  __device__ __forceinline__ double T() const { return phi[s]; }
  __device__ __forceinline__ double S() const { return phi[ld + s]; }
  __device__ __forceinline__ double par() const { return param[s]; }
  __device__ __forceinline__ double n(int k) const { return phi[(int64_t)(k + 2) * ld + s]; }
};

// dPhi/dt of a batch; accumulators in the block's workspace [ns][32].
struct SourceOut {
  double* __restrict__ out;
  double* __restrict__ ws;  // this lane's column
  int64_t ld, s;
  int ns;
  int* status;
  __device__ __forceinline__ double* acc(int k) const { return ws + k * kTile; }
  __device__ __forceinline__ void species(int k, double V, double wk) const {
    if (k < ns - 1) out[(int64_t)(k + 2) * ld + s] = V * wk;
  }
  __device__ __forceinline__ void head(double Tdot, double Sdot) const {
    out[s] = Tdot;
    out[ld + s] = Sdot;
  }
  __device__ __forceinline__ void invalid() const {
    write_nan_state(out, ld, s, ns + 1);
    if (status) atomicAdd(status, 1);
  }
};

// y = (wdot, dT/dt) of a batch; the production rates accumulate in y itself.
struct YOut {
  double* __restrict__ y;
  int64_t ld, s;
  int ns;
  int* status;
  __device__ __forceinline__ double* acc(int k) const { return y + (int64_t)k * ld + s; }
  __device__ __forceinline__ void species(int, double, double) const {}
  __device__ __forceinline__ void head(double Tdot, double) const { y[(int64_t)ns * ld + s] = Tdot; }
  __device__ __forceinline__ void invalid() const {
    write_nan_state(y, ld, s, ns + 1);
    if (status) atomicAdd(status, 1);
  }
};

}  // namespace pj
