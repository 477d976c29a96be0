"""Step graphs that live through loads: after graph steps the state is changed
through the public calls in ways that keep the allocations (other contents of
the same count, a record in cell order and a shuffled one, fewer particles, one
species only, new fields on a solved step), and the steps that follow agree with
a fresh context's on the same state, which has no graph to replay.

Both contexts run the same kernels on the same state bit for bit; the deposit's
atomics (and, in 3D, the order within a cell) make their sums differ in the last
bits. The bounds are those of the graph tests: FP32 fields 2e-5 of the largest
entry and momenta 2e-5, positions 1e-4, FP64 1e-11; iteration counts within one
(FP64 the same)."""
import numpy as np
import pytest

from relsim_inputs import random_state, random_state3

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


FORMS = {"2d": ((24, 16), 32, {}), "2d64": ((24, 16), 64, {}), "launches": ((24, 16), 32, dict(gmres_maxit=(1 << 20) + 1)),
         "quad": ((20, 12), 32, dict(shape=2)), "3d": ((12, 8, 6), 32, {})}


def make(rs, form, stream=None):
    dims, prec, kw = FORMS[form]
    kw = dict(kw, nz=dims[2]) if len(dims) == 3 else kw
    return rs.Simulation(rs.make_config(dims[0], dims[1], dt=0.4, precision=prec, track_ids=True,
                                        gmres_tol=1e-12 if prec == 64 else 1e-7, **kw), stream)


def state(form, seed, counts=(3000, 2600)):
    dims = FORMS[form][0]
    fn = random_state if len(dims) == 2 else random_state3
    return fn(*dims, list(counts), seed=seed, u_scale=0.5, field_scale=0.2)


def record(sp, order):
    at = [sp[k][order] for k in "xyz" if k in sp]
    return np.stack(at, axis=1), np.stack([sp[k][order] for k in ("ux", "uy", "uz")], axis=1), sp["w"][order]


def by_cell(dims, sp):
    key = 0
    for k, L in reversed(list(zip("xyz", dims))):
        key = key * L + np.floor(sp[k])
    return np.argsort(key, kind="stable")


def change(sim, form, how):
    """One change through the public calls."""
    dims = FORMS[form][0]
    st = state(form, 77)
    if how in ("same count", "fewer"):
        if how == "fewer":
            st = state(form, 78, (1700, 900))
        sim.load_state(st)
    elif how in ("in cell order", "shuffled"):
        for s, sp in enumerate(st["species"]):
            order = by_cell(dims, sp) if how == "in cell order" else np.random.default_rng(s).permutation(len(sp["w"]))
            sim.load_species(s, *record(sp, order))
        sim.set_fields(st["E"], st["B"])
    elif how == "one species":
        sim.load_species(1, *record(st["species"][1], slice(None)))
    else:   # "fields on a solved step"
        sim.build()
        sim.solve()
        sim.set_fields(st["E"], st["B"])


def copy_state(sim, to):
    """The state as it is, bit for bit, into a fresh context."""
    for s in range(2):
        start, off, u, w, ids = sim.particles_native(s, ids=True)
        to.load_species_native(s, start, off, u, w, ids)
    to.set_fields(*sim.fields())


def agree(rs, form, a, b, its):
    dims, prec, _ = FORMS[form]
    tol, tx = (1e-11, 1e-11) if prec == 64 else (2e-5, 1e-4)
    assert all(abs(x - y) <= (0 if prec == 64 else 1) for x, y in its), its
    for x, y in zip(a.fields(), b.fields()):
        assert np.abs(x - y).max() <= tol * np.abs(y).max()
    L = np.array(dims, float)
    for s in range(2):
        xa, ua, wa, ia = a.particles(s, ids=True)
        xb, ub, wb, ib = b.particles(s, ids=True)
        oa, ob = np.argsort(ia), np.argsort(ib)
        assert np.array_equal(wa[oa], wb[ob])
        assert np.abs(ua[oa] - ub[ob]).max() <= tol * np.abs(ub).max()
        d = np.abs(xa[oa] - xb[ob])
        assert np.minimum(d, L - d).max() <= tx
    la, lb = a.ledger(), b.ledger()
    for k in ("W_E", "W_B", "K", "dW_E", "dW_B", "dK", "work_grid"):
        assert abs(la[k] - lb[k]) <= tol * lb["total"], k


CHANGES = ("same count", "in cell order", "shuffled", "fewer", "one species", "fields on a solved step")


@pytest.mark.parametrize("form", list(FORMS))
def test_steps_after_a_change_of_state(rs, form):
    sim = make(rs, form)
    sim.load_state(state(form, 5))
    graphs = 0
    for how in CHANGES + CHANGES[::-1]:
        for _ in range(3):
            _, code = sim.step()
            assert code == 0
        change(sim, form, how)
        fresh = make(rs, form)
        copy_state(sim, fresh)
        its = []
        for _ in range(3):
            (la, ca), (lb, cb) = sim.step(), fresh.step()
            assert ca == cb == 0
            its.append((la["gmres_iters"], lb["gmres_iters"]))
        info = sim.graph_info()
        assert not info["disabled"], info["why"]
        assert info["graph_steps"] > graphs
        graphs = info["graph_steps"]
        agree(rs, form, sim, fresh, its)
        fresh.close()
    sim.close()


@pytest.mark.parametrize("shared", [True, False])
def test_batch_after_a_change_of_one_instance(rs, shared):
    import torch
    streams = [torch.cuda.Stream() for _ in range(3)]
    sims = [make(rs, "2d", st.cuda_stream) for st in streams]
    for k, sim in enumerate(sims):
        sim.load_state(state("2d", 10 + k))
    batch = rs.Batch(sims, nworkers=3, shared=shared)
    for how in CHANGES:
        _, status, _ = batch.run(3, component=1, nmodes=2)
        assert list(status) == [0, 0, 0]
        change(sims[1], "2d", how)
        fresh = [make(rs, "2d") for _ in sims]
        for a, b in zip(sims, fresh):
            copy_state(a, b)
        for n in (1, 2):   # the changed instance's first step is host-driven, so the others' is no shared one
            _, status, _ = batch.run(n, component=1, nmodes=2)
            assert list(status) == [0, 0, 0]
        assert batch.last_path == ("shared" if shared else "graphs")
        for a, b in zip(sims, fresh):
            for _ in range(3):
                assert b.step()[1] == 0
            agree(rs, "2d", a, b, [])
            b.close()
    batch.close()
    for sim in sims:
        sim.close()
