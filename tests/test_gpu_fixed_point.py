"""The fixed-point rate constants at the edges of their range: temperatures
around 128 K (below it states take the FP64 path), cold and hot states, and
mechanisms whose constants the fixed point cannot hold (every state on the
FP64 path), against the oracle at the parity tolerances."""
import numpy as np
import pytest

import oracle
import synth
from tests import tiny_mechs as tm
from tests.parity import RTOL_SRC, ATOL_SRC, RTOL_JAC, ATOL_JAC, check_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pj():
    import paper_1809_01029_gb300 as pj
    from paper_1809_01029_gb300 import build
    build.build()
    pj.load_library()
    return pj


def _mech(mechs, name):
    m = (getattr(tm, name)() if name in ("all_kinds", "all_types") else mechs(name)).copy()
    return m


def _compare(pj, m, mode, n, seed, T_range, what):
    import torch
    h = pj.pj_mech_create(m)
    phi, par = synth.make_states(m, n, seed, mode, T_range=T_range)
    if T_range[0] < 128.0 < T_range[1]:
        T = np.array([128.0, np.nextafter(128.0, 0.0), np.nextafter(128.0, 200.0)])
        phi[2:, :3] *= phi[0, :3] / T  # the same mole fractions at the new temperature
        phi[0, :3] = T
    d_phi, d_par = torch.from_numpy(phi).cuda(), torch.from_numpy(par).cuda()
    f_ref, f_env = oracle.source_term_envelope(m, mode, phi, par)
    J, J_env = oracle.jacobian_envelope(m, mode, phi, par)
    assert np.isfinite(f_ref).all() and np.isfinite(J).all()
    check_close(pj.source_terms(h, mode, d_phi, d_par).cpu().numpy(), f_ref, f_env, RTOL_SRC, ATOL_SRC, what)
    dphi = torch.empty_like(d_phi)
    vals = pj.jacobian_sparse(h, mode, d_phi, d_par, dphi=dphi).cpu().numpy()
    check_close(dphi.cpu().numpy(), f_ref, f_env, RTOL_SRC, ATOL_SRC, what + " (jacobian kernel)")
    check_close(vals, oracle.dense_to_csr_values(m, J), oracle.dense_to_csr_values(m, J_env), RTOL_JAC, ATOL_JAC,
                what + " CSR")


@pytest.mark.parametrize("mode", [synth.CONP, synth.CONV])
@pytest.mark.parametrize("T_range", [(100.0, 160.0), (240.0, 400.0), (3000.0, 6000.0)])
@pytest.mark.parametrize("name", ["all_kinds", "all_types", "h2co13"])
def test_temperature_range(pj, mechs, name, T_range, mode):
    _compare(pj, _mech(mechs, name), mode, 45, 61, T_range, f"{name} {T_range} mode={mode}")


@pytest.mark.parametrize("field,value", [("Ea", 2.0e5), ("beta", 90.0), ("Ea0", -1.9e5)])
def test_constants_beyond_the_fixed_point(pj, mechs, field, value):
    """A rate constant outside the fixed point's range (the factor it adds is
    taken out of A, so that rates stay finite)."""
    m = _mech(mechs, "all_kinds")
    i = 6 if field.endswith("0") else 0
    a = "A0" if field.endswith("0") else "A"
    getattr(m, field)[i] = value
    if field == "beta":
        getattr(m, a)[i] *= 1500.0 ** -value
    else:
        getattr(m, a)[i] *= np.exp(value / (1.98720425864083 * 1500.0))
    _compare(pj, m, synth.CONP, 40, 62, (1300.0, 1700.0), f"{field}={value}")
