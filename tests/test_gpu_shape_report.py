"""lbm_get_info: the launch shapes chosen, and in step_threads the block of the even steps as they
run -- pairs of cells in blocks of 128 in shapes 6-10, one plane per thread in blocks of 128 where
no shape was set and there are no pairs (contexts too small for them, full-way walls, the box)."""
import pytest

pytestmark = pytest.mark.gpu


def _lattice(lbm, prec, wall="halfway", geometry="pipe", side=22, nz=9, R=9.3):
    return lbm.Lattice(lbm.make_grid(side, side, nz, R if geometry == "pipe" else 0.0, geometry=geometry, precision=prec,
                                     wall=wall), lbm.lbm_relax(1.5), lbm.make_force(g=(0, 0, 1e-5)))


def _shapes(L):
    i = L.info()
    return i["variant"], i["variant_odd"], i["step_threads"]


@pytest.mark.parametrize("prec", ["f32", "f16s", "bf16"])
@pytest.mark.parametrize("wall,geometry", [("halfway", "pipe"), ("bouzidi", "pipe"), ("fullway", "pipe"), ("halfway", "box")])
def test_default_of_small_and_dense_contexts(lbm_lib, prec, wall, geometry):
    L = _lattice(lbm_lib, prec, wall, geometry)
    assert _shapes(L) == (6 if prec == "f32" and wall != "bouzidi" else 7, 9, 128)
    lbm_lib.lbm_set_variants(L.ctx, 6, 9)
    assert _shapes(L) == (6, 9, 128)
    L.close()


@pytest.mark.parametrize("prec,even,odd", [("f32", 6, 9), ("f16s", 7, 9)])
def test_default_of_a_pipe_on_pairs(lbm_lib, prec, even, odd):
    L = _lattice(lbm_lib, prec, side=44, nz=64, R=20.0)
    assert _shapes(L) == (even, odd, 128)
    L.close()


@pytest.mark.parametrize("shape", range(13))
def test_threads_of_a_set_shape(lbm_lib, shape):
    lbm = lbm_lib
    threads = {0: 256, 1: 256, 2: 128, 3: 512, 4: 256, 5: 128, 11: 992, 12: 512}
    L = _lattice(lbm, "f32")
    lbm.lbm_set_variant(L.ctx, shape)
    assert _shapes(L) == (shape, shape, threads.get(shape, 128))      # pairs: even steps 128
    L.close()
    if shape < 11:
        L = _lattice(lbm, "f32", "fullway")
        lbm.lbm_set_variant(L.ctx, shape)
        assert _shapes(L) == (shape, shape, 256 if shape == 8 else threads.get(shape, 128))
        L.close()
