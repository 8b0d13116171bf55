"""Sides with coefficients above 2: as reactant, as reversible and as
irreversible product, with a third body, in falloff, of the bath gas, first and
last in the mechanism, through every entry point against the oracle; and each
reaction as a mechanism of its own, so that none hides behind a faster one."""
import numpy as np
import pytest

import oracle
import synth
from synth import THIRD_BODY, TROE
from tests import tiny_mechs as tm
from tests.parity import (RTOL_SRC, ATOL_SRC, RTOL_JAC, ATOL_JAC, check_close, jacobian_layout, newton_tol,
                          y_envelope)
from tests.test_gpu_forms import RTOL_VJP

pytestmark = pytest.mark.gpu
U = 2.0 ** -53
H, O, H2, O2, OH, H2O, HO2, N, NO, N2 = range(10)


@pytest.fixture(scope="module")
def pj():
    import paper_1809_01029_gb300 as pj
    from paper_1809_01029_gb300 import build
    build.build()
    pj.load_library()
    return pj


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def mechanism(only=None):
    """Arbitrary (non-physical) parameters; only: the reaction of that index."""
    rx = [
        dict(reac=[(O, 3)], prod=[(H, 1), (HO2, 1)], A=2.0e9, Ea=3000.0, rev=False),
        dict(reac=[(H, 1), (O2, 1)], prod=[(OH, 3)], A=2.0e11, beta=-0.3, Ea=15000.0),
        dict(reac=[(H2, 1)], prod=[(N, 3)], A=4.0e6, beta=0.5, Ea=6000.0),
        dict(reac=[(H, 3)], prod=[(HO2, 1)], A=5.0e9, beta=0.4, kind=TROE, A0=6.0e12, beta0=-0.7, Ea0=500.0,
             troe=(0.7, 90.0, 1800.0, 5000.0), eff={H2: 2.0, H2O: 6.0}),
        dict(reac=[(OH, 3)], prod=[(H2O, 1), (O2, 1)], A=1.5e10, beta=-0.5, kind=THIRD_BODY, eff={H2: 0.7, N2: 1.5}),
        dict(reac=[(O, 1), (H, 1)], prod=[(H2O, 3)], A=3.0e9, rev=False),
        dict(reac=[(N, 3)], prod=[(NO, 3)], A=3.0e8, beta=0.2, Ea=400.0),
        dict(reac=[(H, 4), (O, 1)], prod=[(OH, 2), (NO, 2)], A=3.0e10, Ea=2000.0),
        dict(reac=[(N2, 3)], prod=[(N, 1), (NO, 1)], A=3.0e8, beta=0.1, Ea=900.0),
        dict(reac=[(H, 1), (OH, 1)], prod=[(N2, 3)], A=3.0e7, Ea=1200.0),
        dict(reac=[(O, 1), (H2, 1)], prod=[(OH, 1), (H, 1)], A=4.0e4, beta=2.5, Ea=6000.0),
        dict(reac=[(NO, 3)], prod=[(N2, 1), (O, 2), (O2, 1)], A=3.0e9, Ea=900.0),
    ]
    return synth.build_mechanism("coefficients", tm.SP, rx if only is None else [rx[only]], seed=15)


N_STATES = 70


def _inputs(mode, only=None):
    m = mechanism(only)
    phi, par = synth.make_states(m, N_STATES, 41, mode)
    return m, phi, par


@pytest.mark.parametrize("mode", [synth.CONP, synth.CONV])
def test_source_terms_and_finite_differences(pj, mode):
    m, phi, par = _inputs(mode)
    h = pj.pj_mech_create(m)
    f_ref, f_env = oracle.source_term_envelope(m, mode, phi, par)
    f = pj.source_terms(h, mode, dev(phi), dev(par)).cpu().numpy()
    check_close(f, f_ref, f_env, RTOL_SRC, ATOL_SRC, f"coefficients source terms mode={mode}")
    check_close(pj.eval_y(h, mode, dev(phi), dev(par)).cpu().numpy(), oracle.outputs_y(m, mode, phi, par),
                y_envelope(m, mode, phi, par), RTOL_SRC, ATOL_SRC, f"coefficients y mode={mode}")
    N1 = m.n_species + 1
    J = pj.jacobian_fd(h, mode, dev(phi), dev(par), fmt=pj.PJ_DENSE).cpu().numpy().reshape(N1, N1, -1)
    Jf, _ = oracle.fd_jacobian(m, mode, phi, par)
    hs = oracle.fd_steps(m, mode, phi, par)
    # (a column is NaN where the step takes the bath gas below zero, as the source terms are)
    bath = np.stack([pj.source_terms(h, mode, dev(phi + hs[j] * (np.arange(N1) == j)[:, None]), dev(par)).cpu().numpy()
                     for j in range(N1)], axis=1)
    assert np.array_equal(np.isnan(J), np.isnan(bath)) and np.isnan(J).mean() < 0.05
    assert np.all((np.abs(J - Jf) <= 2 * 4096 * U * f_env[:, None, :] / hs[None, :, :]) | np.isnan(J))


@pytest.mark.parametrize("only", range(12))
def test_each_reaction_alone(pj, only):
    mode = synth.CONP
    m, phi, par = _inputs(mode, only)
    h = pj.pj_mech_create(m)
    J, env = oracle.jacobian_envelope(m, mode, phi, par)
    f_ref, f_env = oracle.source_term_envelope(m, mode, phi, par)
    check_close(pj.source_terms(h, mode, dev(phi), dev(par)).cpu().numpy(), f_ref, f_env, RTOL_SRC, ATOL_SRC,
                f"coefficients reaction {only} source terms")
    check_close(pj.jacobian_sparse(h, mode, dev(phi), dev(par)).cpu().numpy(), oracle.dense_to_csr_values(m, J),
                oracle.dense_to_csr_values(m, env), RTOL_JAC, ATOL_JAC, f"coefficients reaction {only} CSR")
    uw, uT = synth.make_cotangents(m.n_species, N_STATES, 41)
    _, g_phi, g_th = (a.cpu().numpy() for a in pj.vjp(h, mode, dev(phi), dev(par), dev(uw), dev(uT)))
    g_ref, th_ref = oracle.vjp(m, mode, phi, par, uw, uT)
    e_phi, e_th = oracle.vjp_envelope(m, mode, phi, par, uw, uT)
    check_close(g_phi, g_ref, e_phi, RTOL_VJP, 1e-300, f"coefficients reaction {only} g_phi")
    check_close(g_th, th_ref, e_th, RTOL_VJP, 1e-300, f"coefficients reaction {only} g_theta")


@pytest.mark.parametrize("layout", ["coop", "coop-global", "percore"])
@pytest.mark.parametrize("mode", [synth.CONP, synth.CONV])
def test_jacobians_and_newton_matrix(pj, mode, layout):
    m, phi, par = _inputs(mode)
    h = pj.pj_mech_create(m)
    N1 = m.n_species + 1
    J, env = oracle.jacobian_envelope(m, mode, phi, par)
    f_ref, f_env = oracle.source_term_envelope(m, mode, phi, par)
    hs = synth.make_step_sizes(N_STATES, 41)
    d_phi, d_par = dev(phi), dev(par)
    dphi = dev(np.zeros_like(phi))
    with jacobian_layout(layout):
        dense = pj.jacobian_dense(h, mode, d_phi, d_par, dphi=dphi).cpu().numpy().reshape(N1, N1, -1)
        csr = pj.jacobian_sparse(h, mode, d_phi, d_par, fmt=pj.PJ_CSR).cpu().numpy()
        csc = pj.jacobian_sparse(h, mode, d_phi, d_par, fmt=pj.PJ_CSC).cpu().numpy()
        M = pj.newton_matrix_f32(h, mode, d_phi, d_par, dev(hs), 1.0, fmt=pj.PJ_CSR).cpu().numpy()
    what = f"coefficients {layout} mode={mode}"
    check_close(dphi.cpu().numpy(), f_ref, f_env, RTOL_SRC, ATOL_SRC, what + " source terms")
    check_close(dense, J, env, RTOL_JAC, ATOL_JAC, what + " dense")
    assert np.all(dense[~oracle.sparsity_pattern(m)] == 0.0)
    check_close(csr, oracle.dense_to_csr_values(m, J), oracle.dense_to_csr_values(m, env), RTOL_JAC, ATOL_JAC,
                what + " CSR")
    check_close(csc, oracle.dense_to_csc_values(m, J), oracle.dense_to_csc_values(m, env), RTOL_JAC, ATOL_JAC,
                what + " CSC")
    keep = np.flatnonzero((hs[None, None, :] * env).max(axis=(0, 1)) < 1e30)  # well inside FP32's range
    assert len(keep) >= N_STATES // 4
    M_ref = -hs * J
    M_ref[np.arange(N1), np.arange(N1)] += 1.0
    M_ref, scale = (oracle.dense_to_csr_values(m, a)[:, keep] for a in (M_ref, np.abs(M_ref) + hs * env))
    assert np.all(np.abs(M.astype(np.float64)[:, keep] - M_ref) <= newton_tol(scale))


@pytest.mark.parametrize("mode", [synth.CONP, synth.CONV])
def test_vjp(pj, mode):
    m, phi, par = _inputs(mode)
    h = pj.pj_mech_create(m)
    uw, uT = synth.make_cotangents(m.n_species, N_STATES, 41)
    y, g_phi, g_th = (a.cpu().numpy() for a in pj.vjp(h, mode, dev(phi), dev(par), dev(uw), dev(uT)))
    g_ref, th_ref = oracle.vjp(m, mode, phi, par, uw, uT)
    e_phi, e_th = oracle.vjp_envelope(m, mode, phi, par, uw, uT)
    check_close(y, oracle.outputs_y(m, mode, phi, par), y_envelope(m, mode, phi, par), RTOL_SRC, ATOL_SRC,
                f"coefficients vjp y mode={mode}")
    check_close(g_phi, g_ref, e_phi, RTOL_VJP, 1e-300, f"coefficients g_phi mode={mode}")
    check_close(g_th, th_ref, e_th, RTOL_VJP, 1e-300, f"coefficients g_theta mode={mode}")


@pytest.mark.parametrize("config", [(512, 1, 1), (256, 2, 0), (64, 1, 1)])
def test_plans(pj, config):
    import torch
    m, phi, par = _inputs(synth.CONP)
    h = pj.pj_mech_create(m)
    J, env = oracle.jacobian_envelope(m, synth.CONP, phi, par)
    cuts = [0, 33, 34, N_STATES]
    batches = [(dev(par[a:b]), dev(phi[:, a:b]), torch.empty((h.nnz, b - a), dtype=torch.float64, device="cuda"),
                dev(np.zeros_like(phi[:, a:b]))) for a, b in zip(cuts, cuts[1:])]
    plan = pj.Plan(h, pj.PJ_OP_JACOBIAN, synth.CONP, batches)
    plan.set_config(*config)
    plan.run()
    got = np.concatenate([b[2].cpu().numpy() for b in batches], axis=1)
    check_close(got, oracle.dense_to_csr_values(m, J), oracle.dense_to_csr_values(m, env), RTOL_JAC, ATOL_JAC,
                f"coefficients plan {config}")
