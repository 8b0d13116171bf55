"""States outside the fixed point's range: by temperature, and by a Gibbs energy
or enthalpy found too large part of the way, beside states within it.  Values
against the oracle, and bit for bit: what a state gives does not depend on the
states that share its tile."""
import numpy as np
import pytest

import oracle
import synth
from tests import tiny_mechs as tm
from tests.parity import RTOL_SRC, ATOL_SRC, RTOL_JAC, ATOL_JAC, check_close, jacobian_layout, y_envelope
from tests.test_gpu_forms import RTOL_VJP

pytestmark = pytest.mark.gpu


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


def _mech(mechs, name):
    if name == "large_gibbs":
        # |g/RT| of one species goes through the range's end (346 with four
        # coefficients a reaction) between 1000 and 1400 K
        m = tm.all_kinds()
        m.nasa_low[tm.H2, 5] = m.nasa_high[tm.H2, 5] = -4.2e5
        return m
    return getattr(tm, name)() if name in ("all_kinds", "all_types") else mechs(name)


def _states(m, n, seed, mode, name):
    return synth.make_states(m, n, seed, mode, T_range=(700.0, 1700.0) if name == "large_gibbs" else (100.0, 160.0))


@pytest.mark.parametrize("mode", [synth.CONP, synth.CONV])
@pytest.mark.parametrize("name", ["large_gibbs"])
def test_large_gibbs_energies_against_oracle(pj, mechs, name, mode):
    import torch
    m = _mech(mechs, name)
    h = pj.pj_mech_create(m)
    n = 70
    phi, par = _states(m, n, 71, mode, name)
    f_ref, f_env = oracle.source_term_envelope(m, mode, phi, par)
    J, J_env = oracle.jacobian_envelope(m, mode, phi, par)
    assert np.isfinite(f_ref).all() and np.isfinite(J).all()
    d_phi, d_par = dev(phi), dev(par)
    check_close(pj.source_terms(h, mode, d_phi, d_par).cpu().numpy(), f_ref, f_env, RTOL_SRC, ATOL_SRC, f"{name}")
    out = torch.empty_like(d_phi)
    pj.Plan(h, pj.PJ_OP_SOURCE, mode, [(d_par, d_phi, out, None)]).run()
    check_close(out.cpu().numpy(), f_ref, f_env, RTOL_SRC, ATOL_SRC, f"{name} plan")
    ref, env = oracle.dense_to_csr_values(m, J), oracle.dense_to_csr_values(m, J_env)
    for layout in ("coop", "percore"):
        with jacobian_layout(layout):
            vals = pj.jacobian_sparse(h, mode, d_phi, d_par).cpu().numpy()
        check_close(vals, ref, env, RTOL_JAC, ATOL_JAC, f"{name} {layout} CSR")
    uw, uT = synth.make_cotangents(m.n_species, n, 71)
    y, g_phi, g_th = (a.cpu().numpy() for a in pj.vjp(h, mode, d_phi, d_par, dev(uw), dev(uT)))
    check_close(y, oracle.outputs_y(m, mode, phi, par), y_envelope(m, mode, phi, par), RTOL_SRC, ATOL_SRC, f"{name} y")
    g_ref, th_ref = oracle.vjp(m, mode, phi, par, uw, uT)
    e_phi, e_th = oracle.vjp_envelope(m, mode, phi, par, uw, uT)
    check_close(g_phi, g_ref, e_phi, RTOL_VJP, 1e-300, f"{name} g_phi")
    check_close(g_th, th_ref, e_th, RTOL_VJP, 1e-300, f"{name} g_theta")


@pytest.mark.parametrize("mode", [synth.CONP, synth.CONV])
@pytest.mark.parametrize("name", ["all_kinds", "all_types", "large_gibbs", "gri53_types"])
def test_bits_do_not_depend_on_tile_mates(pj, mechs, name, mode):
    """The states of two batches, in tiles of their own and mixed into each
    other's tiles: one batch within the range, the other (cold, or through the
    range's end) not."""
    m = _mech(mechs, name)
    h = pj.pj_mech_create(m)
    n = 64
    a = synth.make_states(m, n, 72, mode, T_range=(1500.0, 2500.0))
    b = _states(m, n, 73, mode, name)
    uw, uT = synth.make_cotangents(m.n_species, n, 74)
    mix = np.arange(n) % 5 == 2

    def outputs(phi, par):
        d_phi, d_par = dev(phi), dev(par)
        y, g_phi, _ = pj.vjp(h, mode, d_phi, d_par, dev(uw), dev(uT))
        return [t.cpu().numpy() for t in (pj.source_terms(h, mode, d_phi, d_par), pj.eval_y(h, mode, d_phi, d_par),
                                          pj.jacobian_fd(h, mode, d_phi, d_par), y, g_phi)]

    of_a, of_b = outputs(*a), outputs(*b)
    of_mix = outputs(np.where(mix, b[0], a[0]), np.where(mix, b[1], a[1]))
    for x, z, got in zip(of_a, of_b, of_mix):
        assert np.array_equal(got, np.where(mix, z, x), equal_nan=True)


def test_a_reaction_outside_leaves_the_others_inside(pj):
    """A reaction whose constants the fixed point cannot hold: the species it
    does not touch keep their production rates bit for bit, and its own agree
    with the oracle (an elementary, a falloff and a third-body reaction)."""
    import torch
    n = 70
    extra = [dict(reac=[(tm.N, 1), (tm.O2, 1)], prod=[(tm.NO, 1), (tm.O, 1)], A=1.0e9, Ea=2.0e5),
             dict(reac=[(tm.NO, 1)], prod=[(tm.N, 1), (tm.O, 1)], A=1.0e9, Ea=1.0e3, kind=synth.TROE, A0=1.0e10, Ea0=-1.9e5,
                  troe=(0.6, 100.0, 1500.0)),
             dict(reac=[(tm.N, 2)], prod=[(tm.N2, 1)], A=1.0e3, beta=101.0, kind=synth.THIRD_BODY, eff={tm.H2: 2.0})]
    base = [dict(reac=[(tm.H, 1), (tm.O2, 1)], prod=[(tm.OH, 1), (tm.O, 1)], A=2.0e11, beta=-0.3, Ea=15000.0),
            dict(reac=[(tm.OH, 2)], prod=[(tm.H2, 1), (tm.HO2, 1)], A=7.0e10, beta=-0.4, kind=synth.TROE, A0=2.0e12,
                 beta0=-0.8, Ea0=-1500.0, troe=(0.7, 90.0, 1800.0, 5000.0), eff={tm.H2O: 6.0}),
            dict(reac=[(tm.H, 1), (tm.OH, 1)], prod=[(tm.H2O, 1)], A=2.0e16, beta=-1.9, kind=synth.THIRD_BODY)]
    for e in extra:  # finite at the batch's temperatures
        e["A"] *= 1500.0 ** -e.get("beta", 0.0) * np.exp(e.get("Ea", 0.0) / (1.98720425864083 * 1500.0))
        if "A0" in e:
            e["A0"] *= np.exp(e["Ea0"] / (1.98720425864083 * 1500.0))
    few, all_ = (synth.build_mechanism("m", tm.SP, rx, seed=21) for rx in (base, base + extra))
    phi, par = synth.make_states(all_, n, 75, synth.CONP, T_range=(1300.0, 1700.0))
    f_ref, f_env = oracle.source_term_envelope(all_, synth.CONP, phi, par)
    J, J_env = oracle.jacobian_envelope(all_, synth.CONP, phi, par)
    assert np.isfinite(f_ref).all() and np.isfinite(J).all()
    y_few, y_all = (pj.eval_y(pj.pj_mech_create(m), synth.CONP, dev(phi), dev(par)) for m in (few, all_))
    untouched = [tm.H, tm.H2, tm.OH, tm.H2O, tm.HO2]
    assert torch.equal(y_few[untouched], y_all[untouched])
    h = pj.pj_mech_create(all_)
    check_close(pj.source_terms(h, synth.CONP, dev(phi), dev(par)).cpu().numpy(), f_ref, f_env, RTOL_SRC, ATOL_SRC, "extra")
    for layout in ("coop", "percore"):
        with jacobian_layout(layout):
            vals = pj.jacobian_sparse(h, synth.CONP, dev(phi), dev(par)).cpu().numpy()
        check_close(vals, oracle.dense_to_csr_values(all_, J), oracle.dense_to_csr_values(all_, J_env), RTOL_JAC, ATOL_JAC,
                    f"extra {layout} CSR")


def test_invalid_state_of_subnormal_temperature(pj):
    """1/T is infinite; the state is invalid and leaves the parameter gradients
    as if it were not there."""
    m = tm.all_kinds()
    h = pj.pj_mech_create(m)
    n = 40
    phi, par = synth.make_states(m, n, 76, synth.CONP)
    uw, uT = synth.make_cotangents(m.n_species, n, 76)
    bad = phi.copy()
    bad[0, 7] = 1e-310
    good = np.arange(n) != 7
    y, g_phi, g_th = (a.cpu().numpy() for a in pj.vjp(h, synth.CONP, dev(bad), dev(par), dev(uw), dev(uT)))
    assert np.isnan(y[:, 7]).all() and np.isnan(g_phi[:, 7]).all()
    _, th_ref = oracle.vjp(m, synth.CONP, phi[:, good], par[good], uw[:, good], uT[good])
    _, e_th = oracle.vjp_envelope(m, synth.CONP, phi[:, good], par[good], uw[:, good], uT[good])
    check_close(g_th, th_ref, e_th, RTOL_VJP, 1e-300, "g_theta beside a state of subnormal temperature")
