"""A force, a force field or a relaxation rate set between replays of a captured chunk holds from
the next step on: the same bytes as direct launches, for one pipe and for an ensemble, in the
kernels that read their member from memory and in those that carry it in the launch parameters
(shapes 6-10).  Both sides run the same kernels on the same numbers: the tolerance is zero.
"""
import pytest

from paper_2405_12082_gb300 import workloads as Wk

pytestmark = pytest.mark.gpu

PIPES = [(22, 21, 9, 9.3), (18, 18, 6, 7.1)]


def _field(p, seed):
    import torch
    nx, ny, nz, _ = p
    return torch.tensor(Wk.gz_field(nz, ny, nx, base=2e-5, seed=seed, rel_amp=0.5), dtype=torch.float32, device="cuda")


def _force(lbm, p, k, field=None):
    trig = Wk.trigger_dict(h=3e-5 * (1 + k), R=p[3], nz=p[2], period=25.0 + k, modes=[(1, 0.6, 0.3), (2, 0.4, 0.0)],
                           t_end=9 + 4 * k)
    return lbm.make_force(g=(1e-6, -2e-6 * k, 3e-5 * (1 + k)), trigger=trig, gz_field=field)


def _run(lbm, chunk, members, prec, wall, shape, change):
    import torch
    pipes = PIPES[:members]
    grids = [lbm.make_grid(*p, precision=prec, wall=wall) for p in pipes]
    forces = [_force(lbm, p, 0) for p in pipes]
    relaxes = [lbm.lbm_relax(1.5) for _ in pipes]
    if members == 1:
        L = lbm.Lattice(grids[0], relaxes[0], forces[0])
    else:
        L = lbm.Lattice(None, None, ensemble=(grids, relaxes, forces))
    if shape is not None:
        lbm.lbm_set_variant(L.ctx, shape)
    lbm.lbm_init(L.ctx, "laminar", noise_amp=4e-3, seed=5)
    lbm.lbm_set_graph(L.ctx, chunk)
    keep = [[_field(p, 3 + k) for k in range(2)] for p in pipes]     # fields of an earlier force stay valid
    L.step(8)
    out = []
    for k in range(2):
        for m, p in enumerate(pipes):
            L.select(m)
            if change == "relax":
                lbm.lbm_set_relax(L.ctx, lbm.lbm_relax(1.7 - 0.2 * k - 0.05 * m))
            else:
                lbm.lbm_set_force(L.ctx, _force(lbm, p, 1 + k + m, keep[m][k] if change == "field" else None))
        L.step(11)                                                   # replays and remainder steps
        L.step(5)
        raw = torch.empty(L.info()["population_bytes"], dtype=torch.uint8, device="cuda")
        lbm.lbm_get_raw(L.ctx, raw, raw.numel())
        out.append(raw)
    L.close()
    return out


@pytest.mark.parametrize("change", ["relax", "force", "field"])
@pytest.mark.parametrize("members", [1, 2])
@pytest.mark.parametrize("prec,wall,shape", [("f32", "halfway", 6), ("f32", "bouzidi", 9), ("f16s", "halfway", 7),
                                             ("bf16", "bouzidi", 10), ("f32", "halfway", None), ("f32", "halfway", 5),
                                             ("f32", "halfway", 11)])
def test_replays_follow_the_setters(lbm_lib, prec, wall, shape, members, change):
    import torch
    direct = _run(lbm_lib, 0, members, prec, wall, shape, change)
    replay = _run(lbm_lib, 4, members, prec, wall, shape, change)
    assert not torch.equal(direct[0], direct[1])
    for a, b in zip(direct, replay):
        assert torch.equal(a, b)


@pytest.mark.parametrize("change", ["field"])
def test_replays_after_an_objective(lbm_lib, change):
    """pipe_objective leaves its force field and omega set: replays after it use them."""
    import torch
    lbm = lbm_lib
    p = PIPES[0]
    out = []
    for chunk in (0, 4):
        L = lbm.Lattice(lbm.make_grid(*p, precision="f32"), lbm.lbm_relax(1.5), lbm.make_force(g=(0, 0, 1e-5)))
        lbm.lbm_set_variants(L.ctx, 6, 9)
        lbm.lbm_init(L.ctx, "laminar", noise_amp=4e-3, seed=5)
        lbm.lbm_set_graph(L.ctx, chunk)
        L.step(8)
        lbm.pipe_objective(L, _field(p, 8), torch.tensor(1.3), 4)
        L.step(12)
        raw = torch.empty(L.info()["population_bytes"], dtype=torch.uint8, device="cuda")
        lbm.lbm_get_raw(L.ctx, raw, raw.numel())
        out.append(raw)
        L.close()
    assert torch.equal(out[0], out[1])
