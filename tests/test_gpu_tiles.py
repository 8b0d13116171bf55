"""The tile kernels at the edges of their launch rules: the source terms' bits
do not depend on the launch shape (16 or 32 warps a tile), the Jacobian's
shapes for mid-size batches agree with the oracle, and the VJP at ragged
tiles, invalid states and states outside the fixed point's range."""
import numpy as np
import pytest

import oracle
import synth
from tests import tiny_mechs as tm
from tests.parity import RTOL_SRC, ATOL_SRC, RTOL_JAC, ATOL_JAC, check_close
from tests.test_gpu_forms import RTOL_VJP, y_envelope

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pj():
    import paper_1809_01029_gb300 as pj
    from paper_1809_01029_gb300 import build
    build.build()
    pj.load_library()
    return pj


def _mech(mechs, name):
    return getattr(tm, name)() if name in ("all_kinds", "bath_efficiency", "all_types") else mechs(name)


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("mode", [synth.CONP, synth.CONV])
@pytest.mark.parametrize("name", ["h2co13", "gri53_types"])
def test_source_terms_bits_do_not_depend_on_the_launch_shape(pj, mechs, name, mode):
    import torch
    m = _mech(mechs, name)
    h = pj.pj_mech_create(m)
    n = 153 * 32 + 7  # more tiles than SMs: 16 warps a tile; the slices: 32
    phi, par = (dev(a) for a in synth.make_states(m, n, 17, mode))
    f, y = pj.source_terms(h, mode, phi, par), pj.eval_y(h, mode, phi, par)
    for lo, hi in ((0, 1), (31, 1000), (4800, n)):
        p = phi[:, lo:hi].contiguous()
        assert torch.equal(pj.source_terms(h, mode, p, par[lo:hi].contiguous()), f[:, lo:hi])
        assert torch.equal(pj.eval_y(h, mode, p, par[lo:hi].contiguous()), y[:, lo:hi])


@pytest.mark.parametrize("name,fmt,n", [("h2co13", "csr", 152 * 512 + 33), ("h2co13", "csc", 152 * 32 + 1),
                                        ("gri53", "dense", 152 * 512 + 5)])
def test_jacobian_of_mid_size_batches(pj, mechs, name, fmt, n):
    """Sampled states of batches on either side of the layout rule's sizes."""
    m = _mech(mechs, name)
    h = pj.pj_mech_create(m)
    phi, par = synth.make_states(m, n, 23, synth.CONV)
    pick = np.unique(np.r_[0, 31, 32, n - 1, np.arange(7, n, n // 20)])
    J, env = oracle.jacobian_envelope(m, synth.CONV, phi[:, pick], par[pick])
    N1 = m.n_species + 1
    if fmt == "dense":
        got = pj.jacobian_dense(h, synth.CONV, dev(phi), dev(par))[:, pick].cpu().numpy().reshape(N1, N1, -1)
    else:
        got = pj.jacobian_sparse(h, synth.CONV, dev(phi), dev(par), fmt=getattr(pj, f"PJ_{fmt.upper()}"))
        got = got[:, pick].cpu().numpy()
        conv = oracle.dense_to_csr_values if fmt == "csr" else oracle.dense_to_csc_values
        J, env = conv(m, J), conv(m, env)
    check_close(got, J, env, RTOL_JAC, ATOL_JAC, f"{name} {fmt} n={n}")


@pytest.mark.parametrize("mode", [synth.CONP, synth.CONV])
@pytest.mark.parametrize("name", ["all_kinds", "all_types", "bath_efficiency"])
def test_vjp_outside_the_fixed_point(pj, mechs, name, mode):
    """States around 128 K: tiles on the general path."""
    m = _mech(mechs, name)
    h = pj.pj_mech_create(m)
    n = 35
    phi, par = synth.make_states(m, n, 29, mode, T_range=(100.0, 160.0))
    uw, uT = synth.make_cotangents(m.n_species, n, 29)
    y, g_phi, g_th = pj.vjp(h, mode, dev(phi), dev(par), dev(uw), dev(uT))
    check_close(y.cpu().numpy(), oracle.outputs_y(m, mode, phi, par), y_envelope(m, mode, phi, par), RTOL_SRC, ATOL_SRC,
                f"{name} cold y")
    g_ref, th_ref = oracle.vjp(m, mode, phi, par, uw, uT)
    e_phi, e_th = oracle.vjp_envelope(m, mode, phi, par, uw, uT)
    check_close(g_phi.cpu().numpy(), g_ref, e_phi, RTOL_VJP, 1e-300, f"{name} cold g_phi")
    check_close(g_th.cpu().numpy(), th_ref, e_th, RTOL_VJP, 1e-300, f"{name} cold g_theta")


@pytest.mark.parametrize("name,n", [("gri53_types", 33), ("h2co13", 700)])
def test_vjp_invalid_states_inside_a_tile(pj, mechs, name, n):
    """Invalid states give NaN and count, and leave the others' gradients and
    the parameter sums as if they were not there."""
    import torch
    m = _mech(mechs, name)
    h = pj.pj_mech_create(m)
    phi, par = synth.make_states(m, n, 31, synth.CONP)
    uw, uT = synth.make_cotangents(m.n_species, n, 31)
    bad = np.array([0, 5, n - 1])
    phi[0, bad[0]], phi[1, bad[1]], phi[2, bad[2]] = -300.0, 0.0, 1e9  # T, V, a bath gas far below zero
    good = np.setdiff1d(np.arange(n), bad)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    y, g_phi, g_th = pj.vjp(h, synth.CONP, dev(phi), dev(par), dev(uw), dev(uT), status=st)
    assert int(st) == len(bad)
    assert torch.isnan(y[:, bad]).all() and torch.isnan(g_phi[:, bad]).all()
    g_ref, th_ref = oracle.vjp(m, synth.CONP, phi[:, good], par[good], uw[:, good], uT[good])
    e_phi, e_th = oracle.vjp_envelope(m, synth.CONP, phi[:, good], par[good], uw[:, good], uT[good])
    check_close(g_phi.cpu().numpy()[:, good], g_ref, e_phi, RTOL_VJP, 1e-300, f"{name} g_phi beside invalid states")
    check_close(g_th.cpu().numpy(), th_ref, e_th, RTOL_VJP, 1e-300, f"{name} g_theta beside invalid states")
