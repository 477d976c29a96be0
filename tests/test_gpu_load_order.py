"""A load finds out in its histogram whether the record lies in cell order, and in
the scan whether a cell is too crowded for the in-cell ordering: one pair out of
order at the edges of warps, blocks and the grid's stride, and cells of 512 and
513 particles, against numpy's stable sort by cell (exact). A record in cell
order takes seven kernels (conversion, histogram, scan in three, kinetic energy
in two)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NX, NY = 16, 12


@pytest.fixture(scope="module")
def rs():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2509_11100_gb300 as rs
    return rs


def record(cells, seed=1):
    r = np.random.default_rng(seed)
    n = len(cells)
    x = np.stack([cells % NX + r.random(n, dtype=np.float32) * 0.5, cells // NX + r.random(n, dtype=np.float32) * 0.5], axis=1)
    return x.astype(np.float64), r.normal(size=(n, 3)).astype(np.float32).astype(np.float64), np.ones(n)


def loaded(rs, cells):
    sim = rs.Simulation(rs.make_config(NX, NY, track_ids=True))
    x, u, w = record(cells)
    n0 = rs.relsim_kernel_launches()
    sim.load_species(0, x, u, w)
    launches = rs.relsim_kernel_launches() - n0
    order = np.argsort(cells, kind="stable")
    _, ug, _, ids = sim.particles(0, ids=True)
    np.testing.assert_array_equal(ids, order)
    np.testing.assert_array_equal(ug, u[order])
    np.testing.assert_array_equal(sim.cell_start(0), np.searchsorted(cells[order], np.arange(NX * NY + 1)))
    sim.close()
    return launches


STRIDE = 152 * 64 * 256   # threads of the largest histogram


@pytest.mark.parametrize("n,at", [(n, at) for n in (2, 33, 5000, STRIDE + 300)
                                  for at in sorted({0, 31, 255, STRIDE - 1, n - 2}) if at <= n - 2])
def test_one_pair_out_of_order(rs, n, at):
    cells = np.sort(np.random.default_rng(3).integers(1, NX * NY - 1, n))
    cells[at + 1:] = np.maximum(cells[at + 1:], 1)
    cells[at + 1] = 0            # below the one before it
    cells[at + 2:] = np.sort(cells[at + 2:])
    loaded(rs, cells)


def test_record_in_cell_order(rs):
    assert loaded(rs, np.sort(np.random.default_rng(3).integers(0, NX * NY, 5000))) == 7


@pytest.mark.parametrize("most", [512, 513])
@pytest.mark.parametrize("cell", [0, 100, NX * NY - 1])
def test_crowded_cell(rs, most, cell):
    r = np.random.default_rng(4)
    others = np.delete(np.arange(NX * NY), cell)
    loaded(rs, r.permutation(np.concatenate([np.full(most, cell), r.choice(others, 2000)])))
