"""lbm_autotune times what lbm_step does: on a small pipe, where a launch that waits for the one
before it costs as much as the step itself, the time it reports is the time of the tuned
context's steps (within 30 %; steps timed apart take 1.6 times as long)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunk", [0, 20])
def test_reported_time_is_that_of_the_steps(lbm_lib, chunk):
    import numpy as np
    import torch
    lbm = lbm_lib
    L = lbm.Lattice(lbm.make_grid(28, 28, 64, 11.5, precision="f32"), lbm.lbm_relax(1.25), lbm.make_force(g=(0, 0, 1e-6)))
    lbm.lbm_init(L.ctx, "laminar", noise_amp=1e-3, seed=2)
    if chunk:
        lbm.lbm_set_graph(L.ctx, chunk)
    f0, f1 = np.empty((27, 64, 28, 28)), np.empty((27, 64, 28, 28))
    lbm.lbm_get_populations(L.ctx, f0)
    shape, us = lbm.lbm_autotune(L.ctx, 200)
    lbm.lbm_get_populations(L.ctx, f1)
    assert np.array_equal(f0, f1) and L.info()["t"] == 0
    assert L.info()["variant"] == shape
    times = []
    for _ in range(7):
        L.step(200)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record()
        L.step(200)
        e1.record()
        torch.cuda.synchronize()
        times.append(1e3 * e0.elapsed_time(e1) / 200)
    step = sorted(times)[3]
    assert step / 1.3 <= us <= 1.3 * step, (us, step, L.info())
    L.close()
