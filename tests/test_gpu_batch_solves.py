"""How a batch's instances solve: where the one-launch solves together want far
more of the GPU than there is, the wide ones (more than a third of it each) go
by launches during the run, the others and every single step do not.

Told from the kernels launched a step: the launches are seven before the first
iteration, three an iteration and five a cycle, where the one-launch solve is
one. The fields agree with those of the same instances stepped one by one within
the bound of the batch tests (1e-4 of the largest entry in FP32; in FP64, where
rounding and the solve's 1e-12 are all that differ, 1e-9)."""
import numpy as np
import pytest

from relsim_inputs import HarrisConfig, make_harris

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


def instances(rs, sizes, precision):
    import torch
    out = []
    for k, (nx, ny) in enumerate(sizes):
        sim = rs.Simulation(rs.make_config(nx, ny, dt=0.5, precision=precision,
                                           gmres_tol=1e-12 if precision == 64 else 1e-7),
                            torch.cuda.Stream().cuda_stream)
        sim.load_state(make_harris(HarrisConfig(nx=nx, ny=ny, ppc=2, dt=0.5, seed=3 + k)))
        out.append(sim)
    return out


WIDE, SMALL = (384, 192), (64, 32)


@pytest.mark.parametrize("precision,sizes,wide", [
    (32, (WIDE, WIDE), 2),
    (32, (WIDE, WIDE, SMALL), 2),
    (32, (WIDE, SMALL), 0),            # together 1.05 of the GPU
    (32, (SMALL, SMALL, SMALL), 0),
    (64, ((128, 64),) * 3, 3),
    (64, ((128, 64), SMALL), 0),
])
def test_batch_solves(rs, precision, sizes, wide):
    steps = 3
    alone, sims = instances(rs, sizes, precision), instances(rs, sizes, precision)
    for sim in alone:
        for _ in range(2):   # the host-driven step, the first graph
            sim.step()
    n0 = rs.relsim_kernel_launches()
    for sim in alone:
        for _ in range(steps):
            sim.step()
    single = rs.relsim_kernel_launches() - n0
    batch = rs.Batch(sims, nworkers=2)
    batch.run(2, nmodes=0)
    n0 = rs.relsim_kernel_launches()
    _, status, iters = batch.run(steps, nmodes=0)
    more = rs.relsim_kernel_launches() - n0 - single
    assert list(status) == [0] * len(sizes)
    assert batch.last_path == "graphs"
    its = int(np.sum(iters[:wide]))
    assert 3 * its + 11 * steps * wide - 3 * wide * steps <= more <= 3 * its + 16 * steps * wide + 3 * wide * steps
    tol = 1e-4 if precision == 32 else 1e-9
    for a, b in zip(alone, sims):
        for fa, fb in zip(a.fields(), b.fields()):
            assert np.max(np.abs(fa - fb)) <= tol * np.abs(fa).max()
    # outside the run a step is in one launch again
    for sims_ in (alone, sims):
        n0 = rs.relsim_kernel_launches()
        for sim in sims_:
            for _ in range(steps):
                sim.step()
        assert rs.relsim_kernel_launches() - n0 == single
    # and a second run goes on as the first
    _, status, _ = batch.run(steps, nmodes=0)
    assert list(status) == [0] * len(sizes)
    batch.close()
    for sim in alone + sims:
        sim.close()
