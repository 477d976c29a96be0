"""A record refused for a non-finite value leaves a state that can be stepped:
the species is as it was, or empty where the record's conversion has taken its
buffer (its particles were loaded in cell order, or the record needs larger
arrays). The refused records have other counts and other cells than the state."""
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


FORMS = {"2d": ((24, 16), {}), "quad": ((20, 12), dict(shape=2)), "3d": ((12, 8, 6), {})}


def records(form, n, seed, in_cell_order=False):
    dims = FORMS[form][0]
    st = (random_state if len(dims) == 2 else random_state3)(*dims, [n, n], seed=seed, u_scale=0.5, field_scale=0.2)
    out = []
    for sp in st["species"]:
        x = np.stack([sp[k] for k in "xyz"[:len(dims)]], axis=1)
        key = 0
        for k in reversed(range(len(dims))):
            key = key * dims[k] + np.floor(x[:, k])
        order = np.argsort(key, kind="stable") if in_cell_order else np.arange(n)
        out.append((x[order], np.stack([sp[k] for k in ("ux", "uy", "uz")], axis=1)[order], sp["w"][order]))
    return out


def refuse(rs, sim, form, n):
    x, u, w = records(form, n, seed=9)[0]
    u[n // 2, 1] = np.nan
    with pytest.raises(rs.RelsimError) as e:
        sim.load_species(0, x, u, w)
    assert e.value.code == rs.RELSIM_ERR_NONFINITE


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("n", [3000, 2100, 3500])   # as many as the state, fewer, more than its arrays hold
@pytest.mark.parametrize("in_cell_order", [False, True])
def test_refused_record(rs, form, n, in_cell_order):
    dims, kw = FORMS[form]
    kw = dict(kw, nz=dims[2]) if len(dims) == 3 else kw
    sim = rs.Simulation(rs.make_config(dims[0], dims[1], dt=0.4, precision=32, track_ids=True, **kw))
    for s, r in enumerate(records(form, 3000, seed=5, in_cell_order=in_cell_order)):
        sim.load_species(s, *r)
    sim.step()   # host-driven
    sim.step()   # and as a graph
    before = [np.array(a) for a in sim.particles(0, ids=True)] + [np.array(sim.cell_start(0))]
    refuse(rs, sim, form, n)
    kept = not in_cell_order and n <= 3000
    assert rs.relsim_num_particles(sim.ctx, 0) == (3000 if kept else 0)
    after = [np.array(a) for a in sim.particles(0, ids=True)] + [np.array(sim.cell_start(0))]
    if kept:
        for a, b in zip(before, after):
            np.testing.assert_array_equal(a, b)
    else:
        assert not after[-1].any()
    for _ in range(2):
        led, status = sim.step()
        assert status == 0 and np.isfinite([v for v in led.values() if isinstance(v, float)]).all()
    ids = np.sort(sim.particles(0, ids=True)[-1])
    np.testing.assert_array_equal(ids, np.arange(3000 if kept else 0))
    np.testing.assert_array_equal(np.sort(sim.particles(1, ids=True)[-1]), np.arange(3000))
    sim.close()


def test_refused_first_record(rs):
    sim = rs.Simulation(rs.make_config(24, 16, dt=0.4, precision=32, track_ids=True))
    sim.load_species(1, *records("2d", 3000, seed=5)[1])
    refuse(rs, sim, "2d", 3000)
    assert rs.relsim_num_particles(sim.ctx, 0) == 0
    led, status = sim.step()
    assert status == 0 and np.isfinite(led["K"])
    sim.close()
