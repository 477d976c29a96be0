"""The counting sort of pushed records (3D and quadratic shapes): one particle,
counts around a block's share of the placement (1024), a species without
particles, moves of several cells, and a second, larger load into the same
context. After a step every particle is once in the cell of its position, with
its own weight bit for bit, and its position, momentum and id belong together:
x' = x + dt u'/gamma'. That sum takes a handful of roundings of values below 8
(positions, moves of up to three cells): 16 of them are 8e-6 in FP32 and 1.5e-14
in FP64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2509_11100_gb300 as rs
    return rs


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("dims", [(7, 5, 3), (7, 6)])
@pytest.mark.parametrize("n", [1, 1023, 1025, 2300])
def test_records_return_to_their_cells(rs, dims, prec, n):
    ft = np.float32 if prec == 32 else np.float64
    D, L, dt = len(dims), np.array(dims, float), 3.0
    kw = dict(nz=dims[2]) if D == 3 else dict(shape=2)
    sim = rs.Simulation(rs.make_config(dims[0], dims[1], dt=dt, precision=prec, track_ids=True, gmres_restart=60,
                                       gmres_maxit=600, gmres_tol=1e-6, **kw))
    nc = int(np.prod(dims))
    for count, seed in ((n, 1), (2 * n + 1, 2)):
        r = np.random.default_rng(seed)
        x0 = np.floor(r.random((count, D)) * L) + (r.integers(0, 2 ** 20, (count, D)) / 2.0 ** 20)
        w0 = (r.random(count) * 1e-3).astype(np.float32).astype(np.float64)
        u0 = r.normal(size=(count, 3)).astype(np.float32).astype(np.float64)
        sim.load_species(0, x0, u0, w0)
        sim.load_species(1, np.zeros((0, D)), np.zeros((0, 3)), np.zeros(0))
        f = (0.1 * r.normal(size=(2, 3, nc))).astype(np.float32).astype(np.float64)
        sim.set_fields(f[0], f[1])
        sim.step()
        start, off, u, w, ids = sim.particles_native(0, ids=True)
        assert start[0] == 0 and start[-1] == count and np.all(np.diff(start) >= 0)
        assert np.array_equal(np.sort(ids), np.arange(count))
        assert np.array_equal(w, w0.astype(ft)[ids])
        cell = np.repeat(np.arange(nc), np.diff(start))
        at = np.stack([cell % dims[0], cell // dims[0] % dims[1], cell // (dims[0] * dims[1])][:D], axis=1)
        assert off.min() >= 0 and off.max() < 1
        u = u.astype(np.float64)
        want = x0[ids] + dt * (u / np.sqrt(1 + (u * u).sum(axis=0))).T[:, :D]
        d = (at + off.T.astype(np.float64) - want + 0.5 * L) % L - 0.5 * L
        assert np.abs(d).max() < (8e-6 if prec == 32 else 1.5e-14)
        assert np.abs(u.T - u0[ids]).max() > 1e-4   # the push has run
    sim.close()
