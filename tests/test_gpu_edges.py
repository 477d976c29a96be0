"""The 3D and quadratic deposits, operators and steps and the load at the edges
of their kernels' units: row segments of one, 32 and 33 cells, odd sizes (the
mass matrix's rows not aligned to 16 bytes), one to four species, empty cells,
cells of one particle and crowded ones, staged batches that end inside a cell;
the load's in-cell ordering at its limit; FP32 values at the ends of their
range through the FP64 record. Tolerances are those of the 3D, quadratic and
load tests (relative to the largest entry)."""
import numpy as np
import pytest

import test_gpu_3d as t3
import test_gpu_quad as tq
from relsim_inputs import random_state, random_state3

pytestmark = pytest.mark.gpu

rs, o3, oq = t3.rs, t3.o3, tq.oq
Q, M = (1.0, -2.0, 0.5, -1.0), (1.0, 3.0, 0.7, 2.0)


def lumpy(st, n, keys, seed):
    """Half of each species' particles moved into two cells' ranges."""
    r = np.random.default_rng(seed)
    for sp in st["species"]:
        pick = r.random(len(sp["w"])) < 0.5
        for k, L in zip(keys, n):
            sp[k] = np.where(pick, (L - 1) * (r.random(len(sp["w"])) < 0.5) + 0.999 * r.random(len(sp["w"])), sp[k])
            sp[k] = np.where(sp[k] >= L, 0.0, sp[k])
    return st


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("n,nsp,per", [((35, 4, 3), 1, 3), ((33, 3, 5), 2, 2), ((64, 3, 3), 4, 1), ((3, 3, 33), 3, 5)])
def test_3d_edges(rs, o3, prec, n, nsp, per):
    nn = n[0] * n[1] * n[2]
    q, m = Q[:nsp], M[:nsp]
    st = t3.f32(lumpy(random_state3(*n, [per * nn + 7 * s for s in range(nsp)], seed=sum(n), u_scale=0.8,
                                    field_scale=0.4, q=q, m=m), n, "xyz", 3))
    sim = t3.sim3(rs, prec, st, dt=0.7, q=q, m=m, nx=n[0], ny=n[1], nz=n[2])
    sim.build()
    Mh, J = sim.mass_matrix()
    c = o3.make_config3(*n, dt=0.7, q=q, m=m, gmres_tol=1e-14, gmres_restart=200)
    P = o3.Particles3(st["species"])
    Jo, Mo = o3.deposit3(c, P, st["B"])
    t = 1e-11 if prec == 64 else 2e-6
    full = t3.full_from_half3(Mh, *n)
    assert t3.rel(J, Jo) < t and t3.rel(full, Mo) < t
    v = np.random.default_rng(4).normal(size=(3, nn))
    assert t3.rel(sim.apply_operator(v), o3.apply_A3(c, full, v)) < (1e-11 if prec == 64 else 1e-5)
    sim.close()


@pytest.mark.parametrize("prec", [64, 32])
def test_3d_step_on_ragged_grid(rs, o3, prec):
    n = (37, 5, 3)
    nn = n[0] * n[1] * n[2]
    st = t3.f32(random_state3(*n, [5 * nn, 4 * nn], seed=8, u_scale=0.5, field_scale=0.2))
    sim = t3.sim3(rs, prec, st, dt=0.5, nx=n[0], ny=n[1], nz=n[2])
    led, code = sim.step()
    assert code == 0
    E, B = sim.fields()
    c = o3.make_config3(*n, dt=0.5, gmres_tol=1e-14, gmres_restart=200)
    P = o3.Particles3(st["species"])
    Eo, Bo, Lo, _ = o3.step3(c, P, st["E"], st["B"])
    tf = 1e-9 if prec == 64 else 2e-5
    assert t3.rel(E, Eo) < tf and t3.rel(B, Bo) < tf
    n0 = P.off[1]
    for s, sl in enumerate((slice(0, n0), slice(n0, None))):
        x, u, w = t3._by_id(sim, s, 0)
        assert t3.rel(u, np.stack([P.ux[sl], P.uy[sl], P.uz[sl]], axis=1)) < tf
        L = np.array(n, float)
        d = (x - np.stack([P.x[sl], P.y[sl], P.z[sl]], axis=1) + 0.5 * L) % L - 0.5 * L
        assert np.abs(d).max() < (1e-10 if prec == 64 else 2e-5)
    total = Lo["W_E1"] + Lo["W_B1"] + Lo["K1"]
    for kg, ko in (("K", "K1"), ("W_E", "W_E1"), ("W_B", "W_B1"), ("work_grid", "work_grid")):
        assert abs(led[kg] - Lo[ko]) < (1e-9 if prec == 64 else 1e-5) * total, kg
    sim.close()


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("n,nsp,per", [((33, 7), 1, 4), ((35, 6), 2, 2), ((64, 5), 4, 1), ((5, 40), 3, 9)])
def test_quadratic_edges(rs, oq, prec, n, nsp, per):
    import oracle
    nn = n[0] * n[1]
    q, m = Q[:nsp], M[:nsp]
    st = tq.f32(lumpy(random_state(*n, [per * nn + 7 * s for s in range(nsp)], seed=sum(n), u_scale=0.8,
                                   field_scale=0.4, q=q, m=m), n, "xy", 3))
    sim = tq.simq(rs, prec, st, *n, dt=0.7, q=q, m=m)
    sim.build()
    Mh, J = sim.mass_matrix()
    c = oracle.make_config(*n, dt=0.7, q=q, m=m)
    Jo, Mo = oq.depositq(c, oracle.Particles(st["species"]), st["B"])
    t = 1e-11 if prec == 64 else 2e-6
    full = tq.full_from_half_q(Mh, *n)
    assert tq.rel(J, Jo) < t and tq.rel(full, Mo) < t
    v = np.random.default_rng(4).normal(size=(3, nn))
    assert tq.rel(sim.apply_operator(v), oq.apply_Aq(c, full, v)) < (1e-11 if prec == 64 else 1e-5)
    sim.close()


@pytest.mark.parametrize("crowd", [511, 512, 513])
def test_load_order_at_the_in_cell_limit(rs, crowd):
    # one cell at, below and above the limit of the in-cell ordering; the
    # load is a stable sort by cell either way
    nx, ny, n = 9, 6, 3000
    r = np.random.default_rng(crowd)
    x = np.stack([r.random(n) * nx, r.random(n) * ny], axis=1)
    inside = (np.floor(x[:, 0]) == 4) & (np.floor(x[:, 1]) == 2)
    x[inside, 0] = 7.5
    x[:crowd] = np.stack([4 + 0.99 * r.random(crowd), 2 + 0.99 * r.random(crowd)], axis=1)
    x = x[r.permutation(n)]
    sim = rs.Simulation(rs.make_config(nx, ny, precision=64, track_ids=True))
    sim.load_species(0, x, r.normal(size=(n, 3)), np.ones(n))
    _, _, _, ids = sim.particles(0, ids=True)
    key = np.floor(x[:, 1]).astype(int) * nx + np.floor(x[:, 0]).astype(int)
    assert np.array_equal(ids, np.argsort(key, kind="stable"))
    assert np.bincount(key, minlength=nx * ny).max() == crowd
    sim.close()


def test_fp32_values_at_the_ends_of_their_range(rs):
    # the record's FP64 values become the FP32 values that a cast gives, and
    # come back as they are: subnormal, tiny, halfway and largest ones
    v = np.array([0.0, -0.0, 1e-45, 1e-40, -3e-39, 2.0 ** -126, 1.0, 1.0 + 2.0 ** -24, 1.0 + 3 * 2.0 ** -24, -1e30,
                  3.0e38, 7e-46, 1.17549429e-38, 0.1])
    n = len(v)
    x = np.stack([np.abs(v) % 1.0 + 1.0, np.linspace(0.0, 2.9, n)], axis=1)
    x[3, 0] = 5e-324
    x[4, 0] = -1e-30
    x[5, 0] = 1e-12
    sim = rs.Simulation(rs.make_config(4, 3, precision=32, track_ids=True))
    sim.load_species(0, x, np.stack([v, v[::-1], -v], axis=1), v)
    xo, uo, wo, ids = sim.particles(0, ids=True)
    back = np.argsort(ids)
    f = v.astype(np.float32).astype(np.float64)
    for got, want in ((wo[back], f), (uo[back][:, 0], f), (uo[back][:, 1], f[::-1]), (uo[back][:, 2], -f)):
        assert np.array_equal(got.view(np.int64), np.ascontiguousarray(want).view(np.int64))
    wrapped = x % np.array([4.0, 3.0])
    wrapped = np.where(wrapped >= np.array([4.0, 3.0]), 0.0, wrapped)   # -1e-30 rounds to the box's length: cell 0
    cell = np.floor(wrapped)
    off = wrapped - cell
    cut = off.astype(np.float32)
    cut = np.where(cut.astype(np.float64) > off, np.nextafter(cut, np.float32(0)), cut).astype(np.float64)
    assert np.array_equal(xo[back], cell + cut)
    sim.close()
