"""Every launch shape on the dense layouts (full-way pipe, periodic box), from even and from odd
t: each steps every fluid cell.  The direct shapes equal shape 2 byte for byte; the pipelined
ones (4, 5) are compiled on their own and agree to the rounding of the steps taken (1e-6 of the
largest population over 5 steps, as on half-way pipes), far below the noise that a cell left out
would keep.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("geometry,wall", [("pipe", "fullway"), ("box", "halfway")])
@pytest.mark.parametrize("prec", ["f32", "f16s"])
@pytest.mark.parametrize("size", [(22, 23, 9, 9.6), (12, 9, 1, 3.2)])
def test_dense_shapes_agree(lbm_lib, geometry, wall, prec, size):
    lbm = lbm_lib
    nx, ny, nz, R = size
    rng = np.random.default_rng(13)
    grid = lbm.make_grid(nx, ny, nz, R if geometry == "pipe" else 0.0, geometry=geometry, precision=prec, wall=wall)
    rho, u = 1 + 0.01 * rng.standard_normal((nz, ny, nx)), 0.02 * rng.standard_normal((3, nz, ny, nx))
    ref = {}
    for shape in [2, 0, 1, 3, 6, 7, 8, 9, 10] + ([4, 5] if prec == "f32" else []):
        L = lbm.Lattice(grid, lbm.lbm_relax(1.4), lbm.make_force(g=(1e-5, -2e-5, 3e-5)))
        lbm.lbm_set_variant(L.ctx, shape)
        lbm.lbm_init_fields(L.ctx, rho, u)
        for steps in (1, 1, 3):
            L.step(steps)
            f = np.empty((27, nz, ny, nx))
            lbm.lbm_get_populations(L.ctx, f)
            t = L.info()["t"]
            if shape == 2:
                ref[t] = f
            elif shape in (4, 5):
                assert np.max(np.abs(f - ref[t])) <= 1e-6 * np.max(np.abs(ref[t])), (shape, t)
            else:
                assert np.array_equal(f, ref[t]), (shape, t)
        L.close()
