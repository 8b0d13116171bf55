"""The LU solve on either side of the rule between its two kernels: both add in
the same order, so a large batch equals its parts bit for bit, in place too."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,dtype,n", [("h2co13", "float64", 152 * 32 + 1), ("h2co13", "float64", 20011),
                                          ("h2co13", "float32", 50001), ("h2co13", "float32", 70007),
                                          ("gri53", "float64", 69999), ("gri53", "float32", 80001)])
def test_solve_of_a_large_batch_equals_its_parts(mechs, name, dtype, n):
    import torch
    import paper_1809_01029_gb300 as pj
    from paper_1809_01029_gb300 import build
    build.build()
    h = pj.pj_mech_create(mechs(name))
    dt = getattr(torch, dtype)
    g = torch.Generator(device="cuda").manual_seed(5)
    lu = 0.1 * torch.randn((h.lu_info()[0], n), dtype=dt, device="cuda", generator=g)
    b = torch.randn((h.n_species + 1, n), dtype=dt, device="cuda", generator=g)
    x = pj.lu_solve(h, lu, b)
    assert torch.isfinite(x).all()
    for lo, hi in ((0, 1), (31, 1000), (n - 777, n)):
        assert torch.equal(pj.lu_solve(h, lu[:, lo:hi].contiguous(), b[:, lo:hi].contiguous()), x[:, lo:hi])
    assert torch.equal(pj.lu_solve(h, lu, b, out=b), x)
