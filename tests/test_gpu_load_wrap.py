"""Loads with finite coordinates far outside the box, up to the largest number:
every particle in the cell and at the offset of the exact remainder (numpy's mod
is exact), sorted and in load order within a cell, in 2D and 3D and both forms."""
import numpy as np
import pytest

import test_gpu_parity as tp

pytestmark = pytest.mark.gpu

rs = tp.rs
FAR = np.array([3.3e25, -3.3e25, 1e17, -1e17, -3e40, 1e300, -1e300, 1.7e308, 2.0 ** 53 + 2, -(2.0 ** 60), 4503599627370497.5,
                -1e-30, -5e-324, 1e-320, 36.999999999, 37.0, -0.25])


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("dims", [(37, 6), (37, 6, 5)])
def test_far_coordinates_land_in_their_cells(rs, prec, dims):
    ft = np.float32 if prec == 32 else np.float64
    r = np.random.default_rng(3)
    n, L = 400, np.array(dims, float)
    x = r.random((n, len(dims))) * L
    for k in range(len(dims)):
        x[r.permutation(n)[:len(FAR)], k] = FAR
    sim = rs.Simulation(rs.make_config(dims[0], dims[1], nz=dims[2] if len(dims) == 3 else None, precision=prec,
                                       track_ids=True))
    sim.load_species(0, x, np.zeros((n, 3)), np.ones(n))
    start, off, _, _, ids = sim.particles_native(0, ids=True)
    at = np.mod(x, L)
    at = np.where(at >= L, 0.0, at)
    cell = np.floor(at)
    key = cell @ np.concatenate([[1.0], np.cumprod(L)[:-1]])
    assert np.array_equal(ids, np.argsort(key, kind="stable"))
    assert np.array_equal(np.diff(start), np.bincount(key.astype(int), minlength=int(np.prod(dims))))
    want = at - cell
    cut = want.astype(ft)
    cut = np.where(cut > want, np.nextafter(cut, ft(0)), cut)   # FP32 offsets are cut, not rounded
    assert np.array_equal(off.T, cut[ids])
    sim.close()
