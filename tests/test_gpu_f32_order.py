"""The F32 step's order of operations, which long F32 runs (and the adjoint's forward pass) add up.

* One even and one odd step of a periodic box against the same arithmetic in NumPy, every
  operation rounded once (fused multiply-adds through FP64 with round-to-odd): the same bytes,
  in every launch shape of one cell per thread.  The pair kernels equal those shapes byte for
  byte (test_gpu_pairs).
* The reciprocal of the density, every mantissa: the bits of the division.
"""
import numpy as np
import pytest

from oracle import lattice

pytestmark = pytest.mark.gpu
F, D = np.float32, np.float64
C = [tuple(int(x) for x in c) for c in lattice.C]
DIR = {c: i for i, c in enumerate(C)}
OPP = [DIR[(-x, -y, -z)] for x, y, z in C]
W = [8 / 27 if i == 0 else 2 / 27 if i < 7 else 1 / 54 if i < 19 else 1 / 216 for i in range(27)]


def _fma(a, b, c):
    p = D(a) * D(b)                                   # exact: 48 bits
    p, c = np.broadcast_arrays(p, D(c))
    s = p + c
    bb = s - p
    e = (p - (s - bb)) + (c - bb)                     # s + e is the exact sum
    bits = s.copy().view(np.int64)
    odd = (e != 0) & ((bits & 1) == 0)
    bits[odd] += np.where((e[odd] > 0) == (s[odd] > 0), 1, -1)
    return bits.view(D).astype(F)


def _step_of_cells(v, g, omega):
    """f* - w of cells v [27][n] (f - w), in the library's order."""
    P, S, M = {}, {}, {}
    for b in range(3):
        for a in range(3):
            ip, im, i0 = DIR[a - 1, b - 1, 1], DIR[a - 1, b - 1, -1], DIR[a - 1, b - 1, 0]
            P[a, b] = v[ip] + v[im]
            S[a, b] = P[a, b] + v[i0]
            M[a, b] = v[ip] - v[im]
    Sa = [S[k, 0] + S[k, 1] + S[k, 2] for k in range(3)]
    Sb = [S[0, k] + S[1, k] + S[2, k] for k in range(3)]
    Da = [M[k, 0] + M[k, 1] + M[k, 2] for k in range(3)]
    drho = Sa[0] + Sa[1] + Sa[2]
    j = [Sa[2] - Sa[0], Sb[2] - Sb[0], Da[0] + Da[1] + Da[2]]
    m4 = (S[2, 2] - S[2, 0]) - (S[0, 2] - S[0, 0])
    m5 = Da[2] - Da[0]
    m6 = (M[0, 2] - M[0, 0]) + (M[1, 2] - M[1, 0]) + (M[2, 2] - M[2, 0])
    m7 = (S[0, 1] + S[2, 1]) - (S[1, 0] + S[1, 2])
    x0 = [v[DIR[-1, k, 0]] + v[DIR[1, k, 0]] for k in (-1, 0, 1)]
    m8 = (x0[0] + x0[1] + x0[2]) - (P[1, 0] + P[1, 1] + P[1, 2])
    rho = F(1) + drho
    ir = F(1) / rho
    hg = [F(0.5) * x for x in g]
    u = [_fma(j[k], ir, hg[k]) for k in range(3)]
    u2 = [x * x for x in u]
    hr = F(0.5) * rho

    def cross(m, k, l):
        return _fma(hr, _fma(g[l], u[k], g[k] * u[l]), _fma(-(rho * u[k]), u[l], m))

    def diag(m, k):
        return _fma(rho, _fma(-g[k], u[k], g[0] * u[0]), _fma(-rho, u2[0] - u2[k], m))

    om1 = F(1) - omega
    a4, a5, a6 = (om1 * s for s in (cross(m4, 0, 1), cross(m5, 0, 2), cross(m6, 1, 2)))
    a7, a8 = om1 * diag(m7, 1), om1 * diag(m8, 2)
    six, third, w = F(1 / 6), F(1 / 3), [F(x) for x in W]
    c12 = _fma(w[1], drho, (a7 + a8) * six)
    c34 = _fma(w[1], drho, _fma(a8, six, -(a7 * third)))
    c56 = _fma(w[1], drho, _fma(a7, six, -(a8 * third)))

    def axis(k, c):
        if c == 0:
            return F(-1.5) * u2[k], hg[k] * (F(-3) * u[k])
        return _fma(F(3), u2[k], F(3 * c) * u[k]), hg[k] * _fma(F(6), u[k], F(3 * c))

    out = np.empty_like(v)
    for i, (cx, cy, cz) in enumerate(C):
        (dx, hx), (dy, hy), (dz, hz) = axis(0, cx), axis(1, cy), axis(2, cz)
        Dxy = _fma(dx, dy, dx + dy)
        A = F(1) + Dxy
        Fxy = _fma(hx, F(1) + dy, hy * (F(1) + dx))
        X = _fma(dz, A + Fxy, _fma(hz, A, Dxy + Fxy))
        wr, wd = w[i] * rho, w[i] * drho
        if i == 0:
            out[i] = _fma(w[0], drho, wr * X)
        elif i <= 6:
            out[i] = _fma(wr, X, c12 if cx else c34 if cy else c56)
        elif i <= 18:
            sign = (cx or 1) * (cy or 1) * (cz or 1)
            out[i] = _fma(wr, X, _fma(F(0.25 * sign), a6 if not cx else a5 if not cy else a4, wd))
        else:
            out[i] = _fma(wr, X, wd)
    return out


@pytest.mark.parametrize("shape", [None, 0, 1, 2, 3, 4, 5])
def test_f32_step_in_its_pinned_order(lbm_lib, shape):
    import torch
    lbm = lbm_lib
    nx, ny, nz = 11, 9, 7
    n, omega = nx * ny * nz, F(1.37)
    g = [F(0.013), F(-0.017), F(0.019)]
    rng = np.random.default_rng(41)
    f = np.array(W)[:, None, None, None] * (1 + 0.1 * rng.standard_normal((27, nz, ny, nx)))
    L = lbm.Lattice(lbm.make_grid(nx, ny, nz, geometry="box", precision="f32"), lbm.lbm_relax(float(omega)),
                    lbm.make_force(g=[float(x) for x in g]))
    if shape is not None:
        lbm.lbm_set_variant(L.ctx, shape)
    L.set_populations(f)
    raw = torch.empty(L.info()["population_bytes"] // 4, dtype=torch.float32, device="cuda")

    def state():
        lbm.lbm_get_raw(L.ctx, raw, raw.numel() * 4)
        return raw.cpu().numpy().reshape(27, -1)[:, :n].copy()

    v = state()
    L.step(1)
    post = _step_of_cells(v, g, omega)
    got = state()
    for i in range(27):
        assert np.array_equal(got[OPP[i]].view(np.int32), post[i].view(np.int32)), i
    # odd step: f_i arrives from x - c_i, f*_i is left at x + c_i
    at = post.reshape(27, nz, ny, nx)
    v = np.stack([np.roll(at[i], C[i][::-1], (0, 1, 2)).ravel() for i in range(27)])
    post = _step_of_cells(v, g, omega).reshape(27, nz, ny, nx)
    L.step(1)
    got = state().reshape(27, nz, ny, nx)
    for i in range(27):
        assert np.array_equal(got[i].view(np.int32), np.roll(post[i], C[i][::-1], (0, 1, 2)).view(np.int32)), i
    L.close()


def test_reciprocal_of_the_density(lbm_lib):
    """rho = 1 + drho takes every float of [1, 2); with jx = 1/2 the velocity is half of 1 / rho."""
    import torch
    lbm = lbm_lib
    L = lbm.Lattice(lbm.make_grid(128, 128, 512, geometry="box", precision="f32"), lbm.lbm_relax(1.25))
    rho = 1 + np.arange(2 ** 23, dtype=np.float64) * 2.0 ** -23
    raw = torch.zeros((27, 2 ** 23), dtype=torch.float32, device="cuda")
    raw[0] = torch.from_numpy(rho - 1.5).float().cuda()
    raw[DIR[1, 0, 0]] = 0.5
    lbm.lbm_set_raw(L.ctx, raw, raw.numel() * 4)
    r, u = (x.cpu().numpy() for x in L.moments())
    assert np.array_equal(r.ravel(), rho.astype(F))
    assert np.array_equal(2 * u[0].ravel(), F(1) / rho.astype(F))
    L.close()
