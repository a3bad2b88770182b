"""lbm_reduce's eight-cell float pairs against FP64 sums of the raw populations.

With u = 2^-24 and S the sum of eight cells' magnitudes, two-sum is exact, each error it hands on
is at most u S, and the k-th addition of those errors rounds by at most k u^2 S: 35 u^2 S over eight
cells, below 2^-42 S (the FP64 sums that follow add less than 2^-45).  A value too large for the
float pairs (1e35) sends its cell to the FP64 path.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CX = (0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1)
CZ = (0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, 1, -1, -1, 1, 1, -1, -1, 1, 1, 1, 1, -1, -1, -1, -1)


@pytest.mark.parametrize("nx,nz,R", [(10, 1, 3.9), (40, 31, 18.3)])
@pytest.mark.parametrize("planted", [0.0, 1e35])
def test_sums_of_the_raw_state(lbm_lib, nx, nz, R, planted):
    import torch
    lbm = lbm_lib
    L = lbm.Lattice(lbm.make_grid(nx, nx, nz, R, precision="f32"), lbm.lbm_relax(1.6), lbm.make_force(g=(1e-6, 0, 2e-5)))
    L.init("laminar", noise_amp=5e-3, seed=4)
    L.step(2)                                        # even t: natural layout
    n = L.info()["population_bytes"] // 4
    raw = torch.empty(n, dtype=torch.float32, device="cuda")
    lbm.lbm_get_raw(L.ctx, raw, 4 * n)
    if planted:
        raw[5 * (n // 27)] = planted                 # direction 5 (+z) of the first fluid cell
        lbm.lbm_set_raw(L.ctx, raw, 4 * n)
    f = raw.double().view(27, -1).cpu().numpy()
    out = lbm.lbm_reduce(L.ctx)
    bound = 2.0 ** -42 * np.abs(f).sum()
    assert abs(out[0] - f.sum()) <= bound
    assert abs(out[1] - (np.array(CX)[:, None] * f).sum()) <= bound
    assert abs(out[3] - (np.array(CZ)[:, None] * f).sum()) <= bound
    assert out[4] == 0
    L.close()
