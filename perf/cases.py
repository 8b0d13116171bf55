"""The workloads this library's speed is measured on: each case is one call (or
the pair of calls) that a reacting-flow code or an implicit integrator makes
through the public entry points, on the synthetic mechanisms and state
distributions of ``synth`` (T ~ U[600, 2500] K, P ~ logU[1, 50] atm, mass
fractions Dirichlet(0.5)), over the sizes such programs use.

``listed`` names the cases, ``draw`` gives more of the same ranges, ``prepare``
makes inputs and buffers, ``run`` makes the call, ``work`` counts what the call
cannot do without, and ``exact`` gives the results in plain float64 torch.
"""
import functools
import math

import numpy as np
import torch

import paper_1809_01029_gb300 as pj
import synth

R = 8314.46261815324          # J / (kmol K)
R_CAL = 1.98720425864083      # cal / (mol K)
P_ATM = 101325.0
CONP, CONV = pj.PJ_CONP, pj.PJ_CONV
FMT = {"csr": pj.PJ_CSR, "csc": pj.PJ_CSC, "dense": pj.PJ_DENSE}
MODE = {"conp": CONP, "conv": CONV}

# largest number of states of a drawn case, by operation and mechanism
CAP = {
    "source": {"h2co13": 1 << 20, "gri53": 1 << 20, "gri53_types": 1 << 18, "usc111": 1 << 18},
    "jacobian": {"h2co13": 1 << 19, "gri53": 1 << 17, "gri53_types": 1 << 17, "usc111": 1 << 15},
    "newton": {"h2co13": 1 << 18, "gri53": 1 << 17, "usc111": 1 << 16},
    "vjp": {"h2co13": 1 << 18, "gri53": 1 << 17, "usc111": 1 << 15},
    "lu": {"h2co13": 1 << 17, "gri53": 1 << 16, "usc111": 1 << 13},
}


def listed():
    return [
        # a zero-dimensional reactor network: few states of a small mechanism,
        # every step waits for the call
        dict(name="source_13sp_64", op="source", mech="h2co13", mode="conp", n=64),
        # one rank's share of a strong-scaled flow solver, an odd cell count
        dict(name="source_53sp_2011_conv", op="source", mech="gri53", mode="conv", n=2011),
        # the explicit chemistry of a large flow field
        dict(name="source_53sp_1m", op="source", mech="gri53", mode="conp", n=1 << 20),
        # a small mechanism's implicit integration: source terms and CSR Jacobian
        dict(name="jac_13sp_4096", op="jacobian", mech="h2co13", mode="conp", fmt="csr", n=4096),
        # the main path: source terms and CSR Jacobian of a methane mechanism
        dict(name="jac_53sp_csr_256k", op="jacobian", mech="gri53", mode="conp", fmt="csr", n=1 << 18),
        # constant volume, dense storage for a dense solver, a ragged cell count
        dict(name="jac_53sp_dense_conv", op="jacobian", mech="gri53", mode="conv", fmt="dense", n=30011),
        # every reaction type (P-log, Chebyshev, chemically activated, explicit
        # reverse), column storage for a direct sparse solver
        dict(name="jac_types_csc_conv", op="jacobian", mech="gri53_types", mode="conv", fmt="csc", n=16411),
        # the FP32 Newton matrix of an implicit integrator, ethylene-sized mechanism
        dict(name="newton_111sp_64k", op="newton", mech="usc111", mode="conp", fmt="csr", n=1 << 16),
        # sensitivity analysis: forward and backward through torch.autograd
        dict(name="vjp_53sp_64k", op="vjp", mech="gri53", mode="conp", n=1 << 16),
        # a large hydrocarbon on uneven patches, one captured graph
        dict(name="plan_874sp_ragged", op="plan", what="jacobian", mech="ic5874", mode="conp", fmt="csr",
             sizes="1024,37,611,1300,129"),
        # the Newton system of an implicit step: factor I - h gamma J and solve
        dict(name="lu_53sp_f64", op="lu", mech="gri53", prec="f64", n=50000),
        # the same in FP32 on the assembled matrix, larger mechanism
        dict(name="lu_111sp_f32", op="lu", mech="usc111", prec="f32", n=8191),
    ]


def draw(rng):
    op = rng.choice(["source", "source", "jacobian", "jacobian", "newton", "vjp", "lu", "plan"])
    mode = rng.choice(["conp", "conv"])
    if op == "plan":
        mech = rng.choice(["gri53", "usc111", "ic5874"])
        hi = {"gri53": 30000, "usc111": 8000, "ic5874": 900}[mech]
        sizes = [int(math.exp(rng.uniform(math.log(17), math.log(hi)))) for _ in range(rng.randint(2, 6))]
        return dict(op=op, what=rng.choice(["source", "jacobian"]), mech=mech, mode=mode,
                    fmt=rng.choice(["csr", "csc"]), sizes=",".join(map(str, sizes)))
    mech = rng.choice(sorted(CAP[op]))
    n = int(math.exp(rng.uniform(math.log(16), math.log(CAP[op][mech]))))
    if op == "lu":
        return dict(op=op, mech=mech, prec=rng.choice(["f64", "f32"]), n=n)
    case = dict(op=op, mech=mech, mode=mode, n=n)
    if op in ("jacobian", "newton"):
        case["fmt"] = rng.choice(["csr", "csc", "dense"])
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _mech(key):
    return synth.make_mechanism(key)


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _states(m, n, mode, g):
    """phi [Ns+1, n], param [n]; Dirichlet(1/2) mass fractions as normalised
    squares of normals (chi-squared with one degree of freedom)."""
    u = torch.rand((2, n), generator=g, device="cuda", dtype=torch.float64)
    T = 600.0 + 1900.0 * u[0]
    P = P_ATM * torch.exp(u[1] * math.log(50.0))
    Y = torch.randn((m.n_species, n), generator=g, device="cuda", dtype=torch.float64).square_()
    Y /= Y.sum(0)
    W = torch.tensor(m.W, device="cuda", dtype=torch.float64)[:, None]
    Y /= W
    Y *= (P / (R * T)) / Y.sum(0)
    V = torch.ones_like(T)
    phi = torch.empty((m.n_species + 1, n), device="cuda", dtype=torch.float64)
    phi[0], phi[1] = T, (V if mode == CONP else P)
    phi[2:] = Y[:-1]
    return phi, (P if mode == CONP else V).contiguous()


def _steps(n, g):
    return torch.exp(torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * math.log(1e4)) * 1e-9


def _sizes(case):
    return [int(s) for s in case["sizes"].split(",")]


def prepare(case, seed):
    m = _mech(case["mech"])
    h = pj.pj_mech_create(m)
    g = _generator(seed)
    op, N = case["op"], m.n_species + 1
    s = dict(op=op, mech=h)
    f64 = dict(device="cuda", dtype=torch.float64)
    if op == "lu":
        _, J, hs, b = _newton_system(case["mech"], case["n"], seed)
        rows, cols = _pattern(case["mech"])
        vals = J[rows, cols].contiguous()
        s["lu"] = torch.empty((h.lu_info()[0], case["n"]), device="cuda", dtype=_dtype(case))
        s["x"] = torch.empty((N, case["n"]), device="cuda", dtype=_dtype(case))
        if case["prec"] == "f64":
            s.update(vals=vals, h=hs, b=b)
        else:
            vals *= -hs
            vals[torch.tensor(rows == cols, device="cuda")] += 1.0
            s.update(vals=vals.float(), h=None, b=b.float())
        return s
    mode = MODE[case["mode"]]
    s["mode"] = mode
    if op == "plan":
        jac = case["what"] == "jacobian"
        s["batches"] = []
        for n in _sizes(case):
            phi, par = _states(m, n, mode, g)
            out = torch.empty((h.nnz if jac else N, n), **f64)
            s["batches"].append((par, phi, out, torch.empty((N, n), **f64) if jac else None))
        s["plan"] = pj.Plan(h, pj.PJ_OP_JACOBIAN if jac else pj.PJ_OP_SOURCE, mode, s["batches"],
                            fmt=FMT[case["fmt"]])
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        s["plan"].capture(side)
        return s
    n = case["n"]
    s["phi"], s["param"] = _states(m, n, mode, g)
    if op == "source":
        s["out"] = torch.empty((N, n), **f64)
    elif op in ("jacobian", "newton"):
        rows = N * N if case["fmt"] == "dense" else h.nnz
        s["fmt"] = FMT[case["fmt"]]
        s["out"] = torch.empty((rows, n), device="cuda", dtype=torch.float32 if op == "newton" else torch.float64)
        s["dphi"] = torch.empty((N, n), **f64)
        if op == "newton":
            s["h"] = _steps(n, g)
    else:
        s["phi"].requires_grad_()
        s["theta"] = torch.from_numpy(np.stack(h.arrhenius(), axis=1)).cuda().requires_grad_()
        s["gy"] = torch.randn((N, n), generator=g, **f64)
    return s


def _dtype(case):
    return torch.float64 if case["prec"] == "f64" else torch.float32


def run(s):
    op = s["op"]
    if op == "source":
        return pj.source_terms(s["mech"], s["mode"], s["phi"], s["param"], out=s["out"])
    if op == "jacobian":
        call = pj.jacobian_dense if s["fmt"] == pj.PJ_DENSE else functools.partial(pj.jacobian_sparse, fmt=s["fmt"])
        call(s["mech"], s["mode"], s["phi"], s["param"], out=s["out"], dphi=s["dphi"])
        return s["out"], s["dphi"]
    if op == "newton":
        pj.newton_matrix_f32(s["mech"], s["mode"], s["phi"], s["param"], s["h"], fmt=s["fmt"], out=s["out"],
                             dphi=s["dphi"])
        return s["out"], s["dphi"]
    if op == "vjp":
        y = pj.source_terms_y(s["mech"], s["mode"], s["phi"], s["param"], s["theta"])
        g_phi, g_theta = torch.autograd.grad(y, (s["phi"], s["theta"]), s["gy"])
        return y, g_phi, g_theta
    if op == "plan":
        s["plan"].launch()
        return [t for _, _, out, dphi in s["batches"] for t in (out, dphi) if t is not None]
    pj.lu_factor(s["mech"], s["vals"], h=s["h"], out=s["lu"])
    pj.lu_solve(s["mech"], s["lu"], s["b"], out=s["x"])
    return s["lu"], s["x"]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
# floating-point operations per state of the method (an exponential 18, a
# logarithm 60, a division 11): source terms, source terms + Jacobian, LU
FLOPS = {
    "h2co13": (3100, 5100, 1200), "gri53": (28800, 48400, 78800), "gri53_types": (29500, 49700, 78800),
    "usc111": (69100, 119000, 644000), "ic5874": (372000, 683000, 0),
}


def work(case):
    m = _mech(case["mech"])
    N, nnz = m.n_species + 1, len(_pattern(case["mech"])[0])
    n = sum(_sizes(case)) if case["op"] == "plan" else case["n"]
    src, jac, lu = FLOPS[case["mech"]]
    states = (N + 1) * 8
    entries = N * N if case.get("fmt") == "dense" else nnz
    if case["op"] == "source" or case.get("what") == "source":
        per, fl = states + N * 8, src
    elif case["op"] in ("jacobian", "plan"):
        per, fl = states + N * 8 + entries * 8, jac
    elif case["op"] == "newton":
        per, fl = states + 8 + N * 8 + entries * 4, jac
    elif case["op"] == "vjp":
        per, fl = states + 3 * N * 8, 2 * src
    else:
        size = 8 if case["prec"] == "f64" else 4
        k = _lu_nnz(case["mech"])
        per, fl = (nnz + k + 2 * N) * size, lu + 2 * k
    return {"bytes": float(per) * n, "flops": float(fl) * n}


@functools.lru_cache(maxsize=None)
def _lu_nnz(key):
    h = pj.pj_mech_create(_mech(key))
    return h.lu_info()[0]


# ---------------------------------------------------------------------------
# the results in plain float64
# ---------------------------------------------------------------------------
FALLOFF = (synth.LINDEMANN, synth.TROE, synth.SRI)


def _net(m, i):
    nu = {}
    for k, v in m.reactants(i):
        nu[k] = nu.get(k, 0) - v
    for k, v in m.products(i):
        nu[k] = nu.get(k, 0) + v
    return {k: v for k, v in nu.items() if v}


@functools.lru_cache(maxsize=None)
def _pattern(key):
    """Row-major (rows, cols) of the Jacobian's fixed pattern: rows and columns
    of T and S, the diagonal, and row k column j where a reaction that changes
    k has a rate depending on n_j."""
    m = _mech(key)
    ns = m.n_species
    mask = np.eye(ns + 1, dtype=bool)
    mask[:2], mask[:, :2] = True, True
    for i in range(m.n_reactions):
        dep = {k for k, _ in m.reactants(i)} | ({k for k, _ in m.products(i)} if m.reversible[i] else set())
        eff = m.efficiencies(i) if m.kind[i] == synth.THIRD_BODY or m.kind[i] in FALLOFF else {}
        dep |= {k for k, a in eff.items() if a != 1.0}
        every = ns - 1 in dep or eff.get(ns - 1, 1.0) != 1.0
        cols = slice(2, None) if every else [j + 2 for j in dep]
        for k in _net(m, i):
            if k < ns - 1:
                mask[k + 2, cols] = True
    return np.nonzero(mask)


def _thermo(m, T):
    """cp/R, h/RT, g/RT and d(cp/R)/dT of every species ([Ns, n], T real or complex)."""
    low = T.real < torch.tensor(m.T_mid, device=T.device)[:, None]
    a = [torch.where(low, torch.tensor(m.nasa_low[:, j], device=T.device)[:, None],
                     torch.tensor(m.nasa_high[:, j], device=T.device)[:, None]) for j in range(7)]
    cp = a[0] + T * (a[1] + T * (a[2] + T * (a[3] + T * a[4])))
    dcp = a[1] + T * (2 * a[2] + T * (3 * a[3] + T * 4 * a[4]))
    h = a[0] + T * (a[1] / 2 + T * (a[2] / 3 + T * (a[3] / 4 + T * a[4] / 5))) + a[5] / T
    s = a[0] * torch.log(T) + T * (a[1] + T * (a[2] / 2 + T * (a[3] / 3 + T * a[4] / 4))) + a[6]
    return cp, h, h - s, dcp


def _arr(A, beta, Ea, T):
    return math.log(A) + beta * torch.log(T) - (Ea / R_CAL) / T


def _lnk_table(m, i, T, P):
    """ln k of a P-log or Chebyshev reaction."""
    x = torch.log(P)
    if m.kind[i] == synth.PLOG:
        tab = m.plog_table(i)
        lk = [_arr(A, b, Ea, T) for _, A, b, Ea in tab]
        lp = [math.log(p) for p in tab[:, 0]]
        out = lk[0] + 0 * x
        for j in range(len(tab) - 1):
            inside = (x.real >= lp[j]) & (x.real < lp[j + 1])
            out = torch.where(inside, lk[j] + (lk[j + 1] - lk[j]) * ((x - lp[j]) / (lp[j + 1] - lp[j])), out)
        return torch.where(x.real >= lp[-1], lk[-1] + 0 * x, out)
    t0, t1, p0, p1 = m.cheb_range[i]
    a = m.cheb_table(i)
    tt = (2 / T - 1 / t0 - 1 / t1) / (1 / t1 - 1 / t0)
    pp = (2 * x - math.log(p0) - math.log(p1)) / (math.log(p1) - math.log(p0))

    def basis(z, k):
        ph = [z * 0 + 1, z]
        while len(ph) < k:
            ph.append(2 * z * ph[-1] - ph[-2])
        return ph[:k]
    bt, bp = basis(tt, a.shape[0]), basis(pp, a.shape[1])
    return math.log(10.0) * sum(a[t, q] * bt[t] * bp[q] for t in range(a.shape[0]) for q in range(a.shape[1]))


def _constants(m, i, T, P, M, g, dl=0.0):
    """kf, kr and the pressure factor c of reaction i; dl is added to the ln k
    of its high-pressure (or only) Arrhenius set."""
    kind = m.kind[i]
    chem = kind in FALLOFF and bool(m.chem[i])
    if kind in (synth.PLOG, synth.CHEB):
        lnk = _lnk_table(m, i, T, P)
    else:
        lninf = _arr(m.A[i], m.beta[i], m.Ea[i], T) + dl
        ln0 = _arr(m.A0[i], m.beta0[i], m.Ea0[i], T) if kind in FALLOFF else None
        lnk = ln0 if chem else lninf
    kf = torch.exp(lnk)
    kr = None
    if m.reversible[i]:
        if m.rev_explicit[i]:
            kr = torch.exp(_arr(*m.rev_arr[i], T))
        else:
            nu = _net(m, i)
            lnKc = sum(nu.values()) * torch.log(P_ATM / (R * T)) - sum(v * g[k] for k, v in nu.items())
            kr = torch.exp(lnk - lnKc)
    c = None
    if kind == synth.THIRD_BODY:
        c = M
    elif kind in FALLOFF:
        Pr = torch.exp(ln0 - lninf) * M
        F = 1.0
        if kind == synth.TROE:
            a, T3, T1, T2 = m.troe[i]
            Fc = (1 - a) * torch.exp(-T / T3) + a * torch.exp(-T / T1)
            if m.troe_n[i] == 4:
                Fc = Fc + torch.exp(-T2 / T)
            L = torch.log(Fc) / math.log(10.0)
            xc = torch.log(Pr) / math.log(10.0) - 0.4 - 0.67 * L
            f1 = xc / (0.75 - 1.27 * L - 0.14 * xc)
            F = torch.exp(math.log(10.0) * L / (1 + f1 * f1))
        elif kind == synth.SRI:
            a, b, cc, d, e = m.sri[i]
            x = torch.log(Pr) / math.log(10.0)
            F = d * torch.exp(torch.log(a * torch.exp(-b / T) + torch.exp(-T / cc)) / (1 + x * x)
                              + e * torch.log(T))
        c = F / (1 + Pr) if chem else F / (1 + 1 / Pr)
    return kf, kr, c


def _product(C, side):
    p = 1.0
    for k, v in side:
        p = p * C[k] ** v
    return p


def _evaluate(m, mode, phi, par, jac=True, u=None):
    """Source terms f [N, n] and, with jac, the dense Jacobian [N, N, n]; with
    u [N, n] the y = (wdot, dT/dt) and its vector-Jacobian products instead."""
    ns, n = m.n_species, phi.shape[1]
    N, b = ns + 1, ns - 1
    T = phi[0]
    V, P = (phi[1], par) if mode == CONP else (par, phi[1])
    Ctot = P / (R * T)
    C = torch.empty((ns, n), device=phi.device, dtype=torch.float64)
    C[:b] = phi[2:] / V
    C[b] = Ctot - C[:b].sum(0)
    cp, h, g, dcp = _thermo(m, T)
    dCbT = -Ctot / T
    dCbS = (Ctot - C[b]) / V if mode == CONP else Ctot / P
    eps = 1e-30
    w = torch.zeros_like(C)
    D = torch.zeros((ns, N, n), device=phi.device, dtype=torch.float64) if jac else None
    Tc = torch.complex(T, eps * T)
    gc = _thermo(m, Tc)[2] if jac else None
    q_lna = []
    for i in range(m.n_reactions):
        reac, prod, nu = m.reactants(i), m.products(i), _net(m, i)
        kind, rev = m.kind[i], bool(m.reversible[i])
        eff = m.efficiencies(i) if kind == synth.THIRD_BODY or kind in FALLOFF else {}
        M = Ctot + sum((a - 1.0) * C[k] for k, a in eff.items()) if kind not in (0, synth.PLOG, synth.CHEB) else Ctot
        kf, kr, c = _constants(m, i, T, P, M, g)
        pf = _product(C, reac)
        pr = _product(C, prod) if rev else 0.0
        Rf = kf * pf
        Rr = kr * pr if rev else torch.zeros_like(Rf)
        Rn = Rf - Rr
        cc = 1.0 if c is None else c
        q = cc * Rn
        for k, v in nu.items():
            w[k] += v * q
        if not jac:
            continue
        dlnA = cc * (Rf if rev and m.rev_explicit[i] else Rn)
        # derivatives of kf, kr, c in T, P and M
        if kind in (0, synth.THIRD_BODY) and not m.rev_explicit[i]:
            lf = (m.beta[i] + (m.Ea[i] / R_CAL) / T) / T
            lr = lf - (sum(v * h[k] for k, v in nu.items()) - sum(nu.values())) / T
            RT = Rf * lf - Rr * lr
            RP = cT = 0.0
            cM = 1.0 if kind == synth.THIRD_BODY else 0.0
        else:
            def part(kfd, krd, step):
                return (kfd.imag * pf - (krd.imag * pr if rev else 0.0)) / step
            kd, rd, cd = _constants(m, i, Tc, torch.complex(P, 0 * P), torch.complex(M, 0 * M), gc)
            RT, cT = part(kd, rd, eps * T), 0.0 if cd is None else cd.imag / (eps * T)
            RP = 0.0
            cM = 1.0 if kind == synth.THIRD_BODY else 0.0
            if kind in (synth.PLOG, synth.CHEB):
                kd, rd, _ = _constants(m, i, torch.complex(T, 0 * T), torch.complex(P, eps * P), M,
                                       g.to(torch.complex128))
                RP = part(kd, rd if rd is None or torch.is_complex(rd) else rd + 0j, eps * P)
            if kind in FALLOFF:
                step = eps * M.abs().clamp_min(1e-300)
                cM = _constants(m, i, T, P, torch.complex(M, step), g)[2].imag / step
                if u is not None:
                    one = torch.complex(torch.zeros_like(T), torch.full_like(T, eps))
                    dlnA = (0.0 if m.chem[i] else dlnA) + Rn * _constants(m, i, T, P, M, g, one)[2].imag / eps
            if kind in (synth.PLOG, synth.CHEB):
                dlnA = torch.zeros_like(q)
        # derivatives in the concentrations (the part of M that is the same
        # for every species cancels in G_j - G_bath)
        G = {}
        for side, k0, sign in ((reac, kf, 1.0), (prod, kr, -1.0)) if rev else ((reac, kf, 1.0),):
            for a, (k, v) in enumerate(side):
                d = sign * cc * k0 * v * C[k] ** (v - 1)
                for e, (k2, v2) in enumerate(side):
                    if e != a:
                        d = d * C[k2] ** v2
                G[k] = G.get(k, 0.0) + d
        ab = eff.get(b, 1.0)
        Gb = G.get(b, 0.0)  # the bath gas as a reactant or product
        dM_T, dM_S = ab * dCbT, ((ab * Ctot - M) / V if mode == CONP else ab * Ctot / P)
        qT = cc * RT + Rn * (cT + cM * dM_T) + Gb * dCbT
        qS = Rn * cM * dM_S + Gb * dCbS
        if mode == CONP:
            qS = qS - sum(d * C[k] / V for k, d in G.items() if k != b)
        else:
            qS = qS + cc * RP
        for k, a in eff.items():
            G[k] = G.get(k, 0.0) + Rn * cM * (a - 1.0)
        base = G.pop(b, None)
        for k, v in nu.items():
            D[k, 0] += v * qT
            D[k, 1] += v * qS
            for j, d in G.items():
                D[k, j + 2] += v * d / V
            if base is not None:
                D[k, 2:] -= v * base / V
        if u is not None:
            q_lna.append((nu, dlnA))
    conp = mode == CONP
    E = R * T * (h if conp else h - 1.0)
    Cx = R * (cp if conp else cp - 1.0)
    den = (C * Cx).sum(0)
    Tdot = -(E * w).sum(0) / den
    wf = torch.tensor(1.0 - m.W / m.W[b], device=phi.device)[:, None]
    Om = (wf * w).sum(0)
    f = torch.empty_like(phi)
    f[0] = Tdot
    f[1] = V * Tdot / T + (R * T * V / P) * Om if conp else P * Tdot / T + R * T * Om
    f[2:] = V * w[:b]
    if not jac:
        return f
    numX = torch.einsum("kn,kxn->xn", E, D)
    numX[0] += (Cx * w).sum(0)
    denX = torch.empty_like(numX)
    denX[0] = R * (C * dcp).sum(0) + Cx[b] * dCbT
    denX[1] = (Cx[b] * Ctot - den) / V if conp else Cx[b] * Ctot / P
    denX[2:] = (Cx[:b] - Cx[b]) / V
    JT = -(numX + Tdot * denX) / den
    if u is not None:
        y = torch.cat([w, Tdot[None]])
        g_phi = torch.einsum("kn,kxn->xn", u[:ns], D) + u[ns] * JT
        lnT, inv = torch.log(T), -1.0 / (R_CAL * T)
        g_theta = torch.empty((m.n_reactions, 3), device=phi.device, dtype=torch.float64)
        for i, (nu, dq) in enumerate(q_lna):
            ub = sum(v * (u[k] - u[ns] * E[k] / den) for k, v in nu.items()) * dq if nu else 0 * dq
            g_theta[i] = torch.stack([ub.sum(), (ub * lnT).sum(), (ub * inv).sum()])
        return y, g_phi, g_theta
    J = torch.empty((N, N, n), device=phi.device, dtype=torch.float64)
    dOm = torch.einsum("kn,kxn->xn", wf.expand(ns, n), D)
    J[0] = JT
    if conp:
        J[1] = V / T * JT + (R * T * V / P) * dOm
        J[1, 0] += -V * Tdot / T ** 2 + (R * V / P) * Om
        J[1, 1] += Tdot / T + (R * T / P) * Om
    else:
        J[1] = P / T * JT + R * T * dOm
        J[1, 0] += -P * Tdot / T ** 2 + R * Om
        J[1, 1] += Tdot / T
    J[2:] = V * D[:b]
    if conp:
        J[2:, 1] += w[:b]
    return f, J


def _newton_system(key, n, seed):
    """phi, dense J [N, N, n], per-state steps h and a right-hand side: h takes
    the fastest diagonal mode from resolved to stiff by four orders."""
    m = _mech(key)
    g = _generator(seed)
    phi, par = _states(m, n, CONP, g)
    u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    z = torch.randn(phi.shape, generator=g, device="cuda", dtype=torch.float64)
    J = _evaluate(m, CONP, phi, par)[1]
    top = torch.diagonal(J).abs().amax(1).clamp_min(1e-30)
    return phi, J, torch.exp(u * math.log(1e4)) / top, 1e-3 * phi * z


def _chunks(m, n):
    step = max(256, int(24e9 / (8 * (m.n_species + 1) ** 2)))
    return [(lo, min(n, lo + step)) for lo in range(0, n, step)]


def _f_and_values(key, fmt, mode, phi, par):
    """f and the Jacobian values in the order of fmt, by chunks of states."""
    m = _mech(key)
    rows, cols = _pattern(key)
    if fmt == "csc":
        at = np.lexsort((rows, cols))
        rows, cols = rows[at], cols[at]
    if fmt == "dense":
        rows, cols = (a.reshape(-1) for a in np.indices((m.n_species + 1,) * 2))
    n = phi.shape[1]
    f = torch.empty_like(phi)
    v = torch.empty((len(rows), n), device=phi.device, dtype=torch.float64)
    r, c = (torch.tensor(a, device=phi.device) for a in (rows, cols))
    for lo, hi in _chunks(m, n):
        f[:, lo:hi], J = _evaluate(m, mode, phi[:, lo:hi].contiguous(), par[lo:hi].contiguous())
        v[:, lo:hi] = J[r, c]
    return f, v, torch.tensor(rows == cols, device=phi.device)


def exact(case, seed):
    key, op = case["mech"], case["op"]
    m = _mech(key)
    g = _generator(seed)
    if op == "lu":
        return _exact_lu(case, seed)
    mode = MODE[case["mode"]]
    if op == "plan":
        got = []
        for n in _sizes(case):
            phi, par = _states(m, n, mode, g)
            if case["what"] == "source":
                got.append(_evaluate(m, mode, phi, par, jac=False))
            else:
                f, v, _ = _f_and_values(key, case["fmt"], mode, phi, par)
                got += [v, f]
        return got
    n = case["n"]
    phi, par = _states(m, n, mode, g)
    if op == "source":
        return _evaluate(m, mode, phi, par, jac=False)
    if op == "vjp":
        gy = torch.randn(phi.shape, generator=g, device="cuda", dtype=torch.float64)
        parts = [_evaluate(m, mode, phi[:, lo:hi].contiguous(), par[lo:hi].contiguous(), u=gy[:, lo:hi].contiguous())
                 for lo, hi in _chunks(m, n)]
        return torch.cat([p[0] for p in parts], 1), torch.cat([p[1] for p in parts], 1), sum(p[2] for p in parts)
    hs = _steps(n, g) if op == "newton" else None
    f, v, diag = _f_and_values(key, case["fmt"], mode, phi, par)
    if op == "newton":
        v *= -hs
        v[diag] += 1.0
    return v, f


def _exact_lu(case, seed):
    key, n = case["mech"], case["n"]
    h = pj.pj_mech_create(_mech(key))
    perm = torch.tensor(np.asarray(h.lu_info()[1]), device="cuda", dtype=torch.long)  # the storage's pivot order
    lr, lc = (torch.tensor(np.asarray(a), device="cuda", dtype=torch.long) for a in h.lu_pattern())
    _, J, hs, b = _newton_system(key, n, seed)
    rows, cols = _pattern(key)
    mask = torch.zeros(J.shape[:2], dtype=torch.bool, device="cuda")
    mask[torch.tensor(rows, device="cuda"), torch.tensor(cols, device="cuda")] = True
    A = J * mask[:, :, None]
    A *= -hs
    torch.diagonal(A).add_(1.0)
    if case["prec"] == "f32":  # the matrix and right-hand side as they were given
        A, b = A.float().double(), b.float().double()
    A = A[perm][:, perm].permute(2, 0, 1).contiguous()
    N = A.shape[1]
    for k in range(N):
        A[:, k + 1:, k] /= A[:, k, k, None]
        if k + 1 < N:
            A[:, k + 1:, k + 1:] -= A[:, k + 1:, k, None] * A[:, None, k, k + 1:]
    y = b[perm].t().contiguous()
    for k in range(1, N):
        y[:, k] -= (A[:, k, :k] * y[:, :k]).sum(1)
    for k in range(N - 1, -1, -1):
        y[:, k] = (y[:, k] - (A[:, k, k + 1:] * y[:, k + 1:]).sum(1)) / A[:, k, k]
    lu = A[:, lr, lc].t().contiguous()
    lu[lr == lc] = 1.0 / lu[lr == lc]
    x = torch.empty_like(b)
    x[perm] = y.t()
    return lu, x
