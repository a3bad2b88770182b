"""lbm_reduce on states that tell FP64 sums from shorter ones, and on values no FP32 sum holds.

* A thread of the reduction takes every 311,296th stored cell (1,216 blocks of 256 threads).  The
  first eight of them hold 1 and then values below half an ulp of 1, chosen so that a second
  float that collects them loses the most, each time downwards: 2^-45 of the sum for a pair of
  floats.  In FP64 the mass passes about 30 roundings of 2^-53 each (a thread's own, 8 levels of
  its block, 5 + 8 of the last one): the bound is 2^-48.
* 3e38 in every cell: FP32 sums of two cells overflow.
* Cells with an infinity or a NaN are counted, once each.
"""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
F = np.float32


def _cells():
    """1 and seven values whose FP32 sum, in this order, loses the most in one direction."""
    seq, lo, lost = [F(1)], F(0), Fraction(0)
    for _ in range(7):
        best = None
        for head in range(64):
            for tail in range(8):
                e = F((2 ** 23 + head * 2 ** 17 + tail) * 2.0 ** -48)      # 24 bits below 2^-24
                s = Fraction(float(lo)) + Fraction(float(e)) - Fraction(float(F(lo + e)))
                if best is None or s > best[0]:
                    best = (s, e)
        lost += best[0]
        lo = F(lo + best[1])
        seq.append(best[1])
    assert all(F(1) + e == F(1) for e in seq[1:])
    return seq, lost / (1 + Fraction(float(lo)))


def _lattice(lbm, nx, nz, R):
    L = lbm.Lattice(lbm.make_grid(nx, nx, nz, R, precision="f32"), lbm.lbm_relax(1.6), lbm.make_force(g=(1e-6, 0, 2e-5)))
    L.init("laminar", noise_amp=5e-3, seed=4)
    return L


def _raw(lbm, L):
    import torch
    raw = torch.empty(L.info()["population_bytes"] // 4, dtype=torch.float32, device="cuda")
    lbm.lbm_get_raw(L.ctx, raw, 4 * raw.numel())
    return raw, (raw.view(27, -1) != 0).any(0)              # padding of the rows is zero


def test_mass_of_adversarial_cells(lbm_lib):
    import torch
    lbm = lbm_lib
    seq, lost = _cells()
    assert lost > Fraction(1, 2 ** 46)                      # what a pair of floats would miss
    L = _lattice(lbm, 84, 500, 40.3)
    raw, fluid = _raw(lbm, L)
    group = torch.arange(fluid.numel(), device="cuda") // 311296
    assert int(group[fluid].max()) >= 7
    table = torch.tensor([float(x) for x in seq] + [0.0] * (1 + int(group.max())), device="cuda")
    raw.view(27, -1)[:] = torch.where(fluid, table[group], torch.zeros((), device="cuda"))
    lbm.lbm_set_raw(L.ctx, raw, 4 * raw.numel())
    exact = 27 * sum(int((fluid & (group == k)).sum()) * Fraction(float(x)) for k, x in enumerate(seq))
    out = lbm.lbm_reduce(L.ctx)
    assert abs(Fraction(out[0]) - exact) <= exact / 2 ** 48
    assert max(abs(x) for x in out[1:4]) <= float(exact) * 2.0 ** -48 and out[4] == 0
    L.close()


def test_sums_beyond_fp32(lbm_lib):
    lbm = lbm_lib
    L = _lattice(lbm, 84, 100, 40.3)
    raw, fluid = _raw(lbm, L)
    n = int(fluid.sum())
    assert n > 400000
    raw.view(27, -1)[5, fluid] = 3e38
    lbm.lbm_set_raw(L.ctx, raw, 4 * raw.numel())
    out = lbm.lbm_reduce(L.ctx)
    for k in (0, 3):
        assert abs(out[k] - n * float(F(3e38))) <= 2.0 ** -42 * n * 3e38
    assert out[4] == 0
    L.close()


@pytest.mark.parametrize("planted", [(float("inf"), 0), (float("-inf"), 13), (float("nan"), 26)])
def test_non_finite_cells_are_counted(lbm_lib, planted):
    import torch
    lbm = lbm_lib
    L = _lattice(lbm, 40, 31, 18.3)
    raw, fluid = _raw(lbm, L)
    at = torch.nonzero(fluid).ravel()[[0, 1, 500, 2000, -1]]
    raw.view(27, -1)[planted[1], at] = planted[0]
    raw.view(27, -1)[3, at[0]] = float("nan")               # twice in one cell
    lbm.lbm_set_raw(L.ctx, raw, 4 * raw.numel())
    assert lbm.lbm_reduce(L.ctx)[4] == 5
    L.close()
