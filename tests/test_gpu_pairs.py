"""The pair kernels (two cells per thread, launch shapes 6-10 on compact pipes) against the
one-cell kernels: the same bytes after even and odd steps, where a pair can go wrong -- one to
five planes (periodic neighbours, a single last plane), rows whose length leaves half a pair,
narrow pipes whose cells are all at the wall, half-way and Bouzidi walls, a per-cell force field
and the trigger, statistics on even and odd samples, one pipe and an ensemble.  Every operation
of the collision is a single rounding in both, so the tolerance is zero.
"""
import pytest

from paper_2405_12082_gb300 import workloads as Wk

pytestmark = pytest.mark.gpu

PIPES = [(9, 8, 1, 2.6), (10, 10, 2, 3.9), (21, 23, 3, 8.3), (40, 41, 4, 18.7), (30, 30, 5, 12.7)]


def _setup(lbm, nx, ny, nz, R, prec, wall, phase=0.3):
    import torch
    trig = Wk.trigger_dict(h=3e-5, R=R, nz=nz, period=25.0, modes=[(1, 0.6, phase), (2, 0.4, 0.0)], t_end=3)
    gz = torch.tensor(Wk.gz_field(nz, ny, nx, base=1e-5, seed=5, rel_amp=0.5), dtype=torch.float32, device="cuda")
    return (lbm.make_grid(nx, ny, nz, R, precision=prec, wall=wall), lbm.lbm_relax(1.7),
            lbm.make_force(g=(1e-6, -2e-6, 3e-5), trigger=trig, gz_field=gz), gz)


def _run(lbm, make, members, shape, every):
    import torch
    L, keep = make()
    lbm.lbm_set_variant(L.ctx, shape)
    lbm.lbm_init(L.ctx, "laminar", noise_amp=4e-3, seed=77)
    lbm.lbm_stats_enable(L.ctx, every)
    out = []
    for steps in (1, 1, 3):
        L.step(steps)
        raw = torch.empty(L.info()["population_bytes"], dtype=torch.uint8, device="cuda")
        lbm.lbm_get_raw(L.ctx, raw, raw.numel())
        out.append(raw)
    for k in range(members):
        L.select(k)
        g = L.grid
        acc = torch.empty((4, g.nz, g.ny, g.nx), dtype=torch.float64, device="cuda")
        lbm.lbm_stats_get(L.ctx, acc)
        out.append(acc)
    assert lbm.lbm_reduce(L.ctx)[4] == 0
    L.close()
    return out


@pytest.mark.parametrize("wall", ["halfway", "bouzidi"])
@pytest.mark.parametrize("prec", ["f32", "f16s", "bf16"])
@pytest.mark.parametrize("pipe", PIPES)
def test_pairs_equal_single_cells(lbm_lib, pipe, prec, wall):
    import torch
    lbm = lbm_lib

    def make():
        s = _setup(lbm, *pipe, prec, wall)
        return lbm.Lattice(*s[:3]), s

    for every in (1, 2):
        ref = _run(lbm, make, 1, 2, every)
        for shape in (6, 7, 8, 9, 10):
            got = _run(lbm, make, 1, shape, every)
            for k, (a, b) in enumerate(zip(got, ref)):
                assert torch.equal(a, b), (shape, every, k)


@pytest.mark.parametrize("prec", ["f32", "bf16"])
def test_pairs_in_an_ensemble(lbm_lib, prec):
    import torch
    lbm = lbm_lib

    def make():
        s = [_setup(lbm, *p, prec, "halfway", phase=0.2 * k) for k, p in enumerate(PIPES)]
        return lbm.Lattice(None, None, ensemble=([x[0] for x in s], [x[1] for x in s], [x[2] for x in s])), s

    ref = _run(lbm, make, len(PIPES), 2, 2)
    for shape in (6, 7, 8, 9, 10):
        for k, (a, b) in enumerate(zip(_run(lbm, make, len(PIPES), shape, 2), ref)):
            assert torch.equal(a, b), (shape, k)
