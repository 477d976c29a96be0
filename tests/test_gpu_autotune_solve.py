"""The autotuner times what a step runs: no operator tile heights on a grid that
is solved in one launch, both on one that is solved by launches (an iteration
limit above 2^20, or its size)."""
import pytest

import test_gpu_parity as tp
from relsim_inputs import random_state

pytestmark = pytest.mark.gpu

rs = tp.rs


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("nx,ny,limit,heights", [(48, 24, 0, 0), (48, 24, (1 << 20) + 1, 2), (288, 288, 0, 2)])
def test_operator_heights_are_tried_where_a_step_uses_them(rs, prec, nx, ny, limit, heights):
    st = random_state(nx, ny, nx * ny * 2, seed=3)
    sim = rs.Simulation(rs.make_config(nx, ny, precision=prec, gmres_maxit=limit))
    sim.load_state(st)
    default, other = (8, 4) if prec == 32 else (4, 2)
    sim.set_launch_shapes(0, 0, other)
    t = sim.autotune()
    assert [rows for rows, _ in t["op_tile_rows"]] == [default, other][:heights]
    assert t["op_rows"] in ((default, other) if heights else (0,))
    _, code = sim.step()
    assert code == 0
    sim.close()
