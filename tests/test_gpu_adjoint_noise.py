"""The FP32 objective from a noisy, decaying start over the full horizon, against the library in FP64
on the same inputs (the other FP32 adjoint tests start from rest, where rounding hardly shows).

u = j (1 / rho) + g / 2 in a flow whose density settles near 1 rounds the reciprocal alike in many
cells: at most 2^-25 of u per step, 6e-5 after 2,000.  The objective is a mean over the run (half
of that), the gradients see it once more through the stored moments: 6e-5.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_noisy_start_against_fp64(lbm_lib):
    import torch
    lbm = lbm_lib
    nx, nz, T = 52, 256, 2000
    rng = np.random.default_rng(6)
    rho = 1 + 1e-3 * rng.standard_normal((nz, nx, nx))
    u = 1e-3 * rng.standard_normal((3, nz, nx, nx))
    u[2] += 0.01
    g = torch.tensor(1e-6 * (0.7 + 0.6 * rng.random((nz, nx, nx))), dtype=torch.float32, device="cuda")
    out = {}
    for prec, dt in (("f32", torch.float32), ("f64", torch.float64)):
        gz, omega = g.detach().to(dt).clone().requires_grad_(True), torch.tensor(1.25, dtype=dt, requires_grad=True)
        L = lbm.Lattice(lbm.make_grid(nx, nx, nz, 24.0, precision=prec), lbm.lbm_relax(1.25))
        lbm.lbm_init_fields(L.ctx, rho, u)
        J = lbm.pipe_objective(L, gz, omega, T)
        J.backward()
        out[prec] = [x.detach().double().cpu().numpy() for x in (J, gz.grad, omega.grad, L.moments()[1])]
        L.close()
    for a, b, tol in zip(out["f32"], out["f64"], (3e-5, 6e-5, 6e-5, 6e-5)):
        assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b)
