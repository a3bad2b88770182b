"""lbm_modes from two host threads, rings of 4,096 and of 2,100 samples (both above 48 KB of dynamic
shared memory, which a kernel has to be allowed first): neither call may fail because of the other,
and each gives the bytes it gives alone."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_rings_of_two_sizes_at_once(lbm_lib):
    import torch
    lbm = lbm_lib
    sizes, out, errors = (4096, 2100), {}, []
    ctx = {}
    for n in sizes:
        L = lbm.Lattice(lbm.make_grid(24, 24, 6, 9.5, precision="f32"), lbm.lbm_relax(1.5), lbm.make_force(g=(0, 0, 1e-5)),
                        stream=torch.cuda.Stream().cuda_stream)
        lbm.lbm_init(L.ctx, "laminar", noise_amp=1e-3, seed=4)
        cfg = lbm.make_modes_cfg(2, (0.7,), n, 8)
        E = np.empty((2, 1, 9))
        lbm.lbm_modes(L.ctx, cfg, E)
        ctx[n], out[n] = (L, cfg), E

    def work(n):
        L, cfg = ctx[n]
        E = np.empty_like(out[n])
        try:
            for _ in range(1500):
                lbm.lbm_modes(L.ctx, cfg, E)
                if not np.array_equal(E, out[n]):
                    raise AssertionError("ring of %d samples: other energies" % n)
        except Exception as e:                       # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(n,)) for n in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for L, _ in ctx.values():
        L.close()
    assert not errors, errors
