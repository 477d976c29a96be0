"""The field solve in one launch (grids whose tiles fit on the GPU at once) at
the edges of its tiles: tile heights 1, 2, 4 and 8, narrow and ragged last
tiles, more blocks than SMs, restarts inside the launch, a zero right-hand
side and a run that stops at its iteration limit."""
import numpy as np
import pytest

from relsim_inputs import random_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    import paper_2509_11100_gb300 as m
    m.lib()
    return m


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


def rel(a, b):
    return np.abs(a - b).max() / np.abs(b).max()


def fp32_state(nx, ny, n, seed):
    st = random_state(nx, ny, n, seed=seed, u_scale=0.7, field_scale=0.3)
    for sp in st["species"]:
        for k in ("x", "y", "ux", "uy", "uz", "w"):
            sp[k] = sp[k].astype(np.float32).astype(np.float64)
        sp["x"] = np.where(sp["x"] >= nx, 0.0, sp["x"])
        sp["y"] = np.where(sp["y"] >= ny, 0.0, sp["y"])
    st["E"] = st["E"].astype(np.float32).astype(np.float64)
    st["B"] = st["B"].astype(np.float32).astype(np.float64)
    return st


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("nx,ny", [(3, 3), (31, 9), (64, 32), (65, 66), (128, 130), (200, 150), (257, 131), (33, 400)])
def test_one_launch_solve_matches_oracle(rs, orc, prec, nx, ny):
    # the bounds of the other field-solve tests: 1e-9 with FP64 and a 1e-12
    # tolerance, 2e-5 with FP32 and a 1e-7 one
    st = fp32_state(nx, ny, nx * ny * 2, seed=nx + ny)
    sim = rs.Simulation(rs.make_config(nx, ny, dt=0.5, precision=prec, gmres_tol=1e-12 if prec == 64 else 1e-7,
                                       gmres_restart=6))
    sim.load_state(st)
    sim.build()
    before = rs.relsim_kernel_launches()
    it, relres, status = sim.solve()
    assert status == 0 and (prec == 32 or it > 6)       # FP64: at least one restart
    assert rs.relsim_kernel_launches() - before <= 6    # right-hand side, solve, field update
    c = orc.make_config(nx, ny, dt=0.5, gmres_tol=1e-13, gmres_restart=50)
    Eo, Bo, _, ex = orc.step(c, orc.Particles(st["species"]), st["E"], st["B"], want_matrices=True)
    t = 1e-9 if prec == 64 else 2e-5
    E1, B1 = sim.fields()
    assert rel(sim.E_theta(), ex["Etheta"]) < t
    assert rel(E1, Eo) < 2 * t and rel(B1, Bo) < t
    sim.close()


@pytest.mark.parametrize("prec", [32, 64])
def test_one_launch_solve_zero_and_limit(rs, prec):
    nx, ny = 40, 21
    sim = rs.Simulation(rs.make_config(nx, ny, precision=prec))
    sim.set_fields(np.zeros((3, nx * ny)), np.zeros((3, nx * ny)))
    sim.build()
    it, relres, status = sim.solve()
    assert (it, relres, status) == (0, 0.0, 0)
    assert not sim.E_theta().any()
    sim.close()
    st = fp32_state(nx, ny, nx * ny * 2, seed=5)
    sim = rs.Simulation(rs.make_config(nx, ny, precision=prec, gmres_tol=1e-14, gmres_restart=4, gmres_maxit=7))
    sim.load_state(st)
    sim.build()
    it, relres, status = sim.solve()
    assert it == 7 and status == rs.RELSIM_ERR_NOT_CONVERGED and 0.0 < relres < 1.0
    sim.close()
