"""Quadratic shapes on grids three cells wide, the narrowest accepted, where a
deposit column's nodes reach past the row's end: the deposit and a step against
the oracle, with the bounds of the quadratic tests."""
import numpy as np
import pytest

import test_gpu_quad as tq
from relsim_inputs import random_state

pytestmark = pytest.mark.gpu

rs, oq = tq.rs, tq.oq


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("n", [(3, 3), (3, 4), (3, 5), (4, 3)])
def test_three_cells_wide(rs, oq, prec, n):
    import oracle
    nn = n[0] * n[1]
    st = tq.f32(random_state(*n, [9 * nn, 6 * nn], seed=sum(n), u_scale=0.5, field_scale=0.2))
    sim = tq.simq(rs, prec, st, *n, dt=0.5)
    sim.build()
    Mh, J = sim.mass_matrix()
    c = oracle.make_config(*n, dt=0.5, gmres_tol=1e-14, gmres_restart=200)
    P = oracle.Particles(st["species"])
    Jo, Mo = oq.depositq(c, P, st["B"])
    t = 1e-11 if prec == 64 else 2e-6
    assert tq.rel(J, Jo) < t and tq.rel(tq.full_from_half_q(Mh, *n), Mo) < t
    _, _, status = sim.solve()
    assert status == 0
    sim.push()
    Eo, Bo, _, _ = oq.stepq(c, P, st["E"], st["B"])
    E, B = sim.fields()
    t = 1e-9 if prec == 64 else 2e-5
    assert tq.rel(E, Eo) < t and tq.rel(B, Bo) < t
    n0 = P.off[1]
    for s, sl in enumerate((slice(0, n0), slice(n0, None))):
        _, u, _, ids = sim.particles(s, ids=True)
        assert tq.rel(u[np.argsort(ids)], np.stack([P.ux[sl], P.uy[sl], P.uz[sl]], axis=1)) < t
    sim.close()
