"""The 2D field solve by launches (operator, reduction, basis update with the
cycle's tail, the loops as conditional nodes in a step graph), which grids take
whose tiles do not fit on the GPU at once. An iteration limit above 2^20 has
small grids take it too: the tests of the solve, the adjoints and the graphs run
on it with their own bounds, and it is compared with the one-launch solve of the
same system. A 288x288 grid takes it by its size."""
import numpy as np
import pytest

import test_gpu_adjoint as ta
import test_gpu_parity as tp
import test_gpu_predictor as tpr
import test_gpu_solve as ts

pytestmark = pytest.mark.gpu

rs, orc = tp.rs, tp.orc
LIMIT = (1 << 20) + 1


class ByLaunches:
    """The package, its contexts' iteration limit above 2^20 where none is given."""

    def __init__(self, rs):
        self.rs = rs

    def __getattr__(self, name):
        return getattr(self.rs, name)

    def make_config(self, *args, **kw):
        c = self.rs.make_config(*args, **kw)
        c.gmres_maxit = c.gmres_maxit or LIMIT
        return c


@pytest.fixture(scope="module")
def ls(rs):
    return ByLaunches(rs)


def solved(rs, cfg, st):
    sim = rs.Simulation(cfg)
    sim.load_state(st)
    sim.build()
    before = rs.relsim_kernel_launches()
    out = sim.solve()
    return sim, out, rs.relsim_kernel_launches() - before


FORMS = [(32, False), (32, True), (64, False)]   # precision, FP64 vectors in the FP32 form


@pytest.mark.parametrize("prec,fp64", FORMS)
@pytest.mark.parametrize("nx,ny", [(3, 3), (31, 9), (65, 66), (128, 130), (257, 131), (33, 400)])
def test_launches_match_oracle_and_one_launch(rs, orc, prec, fp64, nx, ny):
    # the grids, restarts and bounds of the one-launch solve's test
    st = ts.fp32_state(nx, ny, nx * ny * 2, seed=nx + ny)
    kw = dict(dt=0.5, precision=prec, gmres_tol=1e-12 if prec == 64 else 1e-7, gmres_restart=6, gmres_fp64=fp64)
    one, (it1, _, status1), few = solved(rs, rs.make_config(nx, ny, **kw), st)
    sim, (it, relres, status), many = solved(rs, rs.make_config(nx, ny, gmres_maxit=LIMIT, **kw), st)
    assert status == status1 == 0 and (prec == 32 or it > 6)
    assert few <= 6 and many > 3 * it   # three kernels an iteration and more
    # the dot products' partial sums add up in another order: an estimate
    # within rounding of the tolerance may stop one iteration apart, and a
    # true residual within rounding of it may take one more
    assert abs(it - it1) <= 2
    c = orc.make_config(nx, ny, dt=0.5, gmres_tol=1e-13, gmres_restart=50)
    Eo, Bo, _, ex = orc.step(c, orc.Particles(st["species"]), st["E"], st["B"], want_matrices=True)
    t = 1e-9 if prec == 64 else 2e-5
    E1, B1 = sim.fields()
    assert ts.rel(sim.E_theta(), ex["Etheta"]) < t
    assert ts.rel(E1, Eo) < 2 * t and ts.rel(B1, Bo) < t
    assert ts.rel(sim.E_theta(), one.E_theta()) < t
    one.close()
    sim.close()


@pytest.mark.parametrize("prec", [32, 64])
def test_zero_right_hand_side(ls, prec):
    nx, ny = 40, 21
    sim = ls.Simulation(ls.make_config(nx, ny, precision=prec))
    sim.set_fields(np.zeros((3, nx * ny)), np.zeros((3, nx * ny)))
    sim.build()
    it, relres, status = sim.solve()
    assert (it, relres, status) == (0, 0.0, 0) and not sim.E_theta().any()
    sim.close()


@pytest.mark.parametrize("prec,fp64", FORMS)
def test_iteration_limit_on_a_large_grid(rs, prec, fp64):
    nx = ny = 288
    st = ts.fp32_state(nx, ny, nx * ny * 2, seed=5)
    sim, (it, relres, status), many = solved(rs, rs.make_config(nx, ny, precision=prec, gmres_tol=1e-14, gmres_restart=4,
                                                                gmres_maxit=7, gmres_fp64=fp64), st)
    assert it == 7 and status == rs.RELSIM_ERR_NOT_CONVERGED and 0.0 < relres < 1.0 and many > 3 * it
    sim.push()
    for _ in range(3):   # host-driven, then graphs
        led, code = sim.step()
        assert code == rs.RELSIM_ERR_NOT_CONVERGED and led["gmres_iters"] == 7 and led["gmres_restarts"] >= 2
    assert sim.graph_info()["graph_steps"] > 0
    sim.close()


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("nx,ny,theta", [(13, 7, 0.5), (24, 16, 0.6)])
def test_field_adjoint(ls, orc, prec, nx, ny, theta):
    ta.test_field_adjoint_matches_oracle(ls, orc, prec, nx, ny, theta)


@pytest.mark.parametrize("prec,fp64", FORMS)
@pytest.mark.parametrize("nx,ny", [(65, 66), (257, 131)])
def test_field_adjoint_with_restarts_matches_one_launch(rs, prec, fp64, nx, ny):
    # both stop at a residual of tol |b| and A's symmetric part is at least
    # one, so the solutions differ by 2 tol |b| at most, all in one entry:
    # 2 tol (3 nx ny)^(1/2) = 640 tol of the largest; the bounds are those of
    # the comparison with the oracle
    st = ts.fp32_state(nx, ny, nx * ny * 2, seed=nx)
    r = np.random.default_rng(2)
    gE, gB = r.normal(size=(3, nx * ny)), r.normal(size=(3, nx * ny))
    tol = 1e-12 if prec == 64 else 1e-7
    out = []
    for limit in (0, LIMIT):
        sim, (_, _, status), _ = solved(rs, rs.make_config(nx, ny, dt=0.5, precision=prec, gmres_tol=tol, gmres_restart=5,
                                                           gmres_maxit=limit, gmres_fp64=fp64), st)
        g = sim.field_adjoint(gE, gB)
        assert status == 0 and g["status"] == 0 and g["iters"] > 5
        out.append(g)
        sim.close()
    assert abs(out[0]["iters"] - out[1]["iters"]) <= 2
    for k in ("E0", "B0", "J", "M"):
        assert ts.rel(out[1][k], out[0][k]) < (1e-9 if prec == 64 else 2e-5), k


@pytest.mark.parametrize("prec", [64, 32])
def test_one_step_adjoint_chain(ls, orc, prec):
    ta.test_one_step_adjoint_chain_matches_oracle(ls, orc, prec)


@pytest.mark.parametrize("prec,pred", [(64, 0), (32, 0), (64, 1), (32, 1)])
def test_step_adjoint(ls, orc, prec, pred):
    ta.test_step_adjoint_in_place_by_id_matches_oracle(ls, orc, prec, pred)


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("theta", [0.5, 0.7])
def test_field_solve(ls, orc, prec, theta):
    tp.test_field_solve_matches_oracle(ls, orc, prec, theta)


@pytest.mark.parametrize("prec", [32, 64])
def test_graph_steps(ls, prec):
    tp.test_graph_steps_match_host_driven_steps(ls, prec)


def test_ten_fp64_steps(ls, orc):
    tp.test_fp64_ten_steps_match_oracle(ls, orc)


def test_predicted_fp64_steps(ls, orc):
    tpr.test_predicted_fp64_steps_match_oracle_and_close_the_ledger(ls, orc)


@pytest.mark.parametrize("case", ["harris", "ragged"])
def test_double_float_krylov(ls, orc, case):
    tp.test_double_float_krylov_matches_fp64_krylov(ls, orc, case)


def test_autotuned_launch_shapes(ls):
    tp.test_autotuned_launch_shapes_give_the_same_steps(ls)


@pytest.mark.parametrize("prec", [32, 64])
def test_operator_tile_heights(ls, prec):
    tp.test_operator_tile_heights_agree(ls, prec)
