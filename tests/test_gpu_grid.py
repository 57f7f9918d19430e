"""Grid density and its adjoint against direct 64-bit sums: supports wider than
the 32-point tiles, supports that reach no point, points on a particle, odd
grids, particle counts around a warp's share, the drift and the periodic wrap."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
GK, KN = 1.825742, 2.5464790894703255


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1807_01341_gb300 import build
    build.build()
    from paper_1807_01341_gb300 import sim
    return torch, sim


def direct(x, m, h, bar, ng):
    rho, grad = np.zeros(ng ** 3), np.zeros((4, len(m)))
    c = (np.arange(ng) + 0.5) / ng
    for j in range(len(m)):
        H = GK * h[j]
        d = [x[j, a] - c for a in range(3)]
        d = [v - np.round(v) for v in d]
        r2 = d[2][:, None, None] ** 2 + d[1][None, :, None] ** 2 + d[0][None, None, :] ** 2
        k = np.nonzero(r2 < H * H)
        r = np.sqrt(r2[k])
        q = r / H
        w = np.where(q < 0.5, 1 - 6 * q ** 2 + 6 * q ** 3, 2 * (1 - q) ** 3)
        dw = np.where(q < 0.5, -12 * q + 18 * q ** 2, -6 * (1 - q) ** 2)
        at = k[2] + ng * (k[1] + ng * k[0])
        rho[at] += m[j] * KN * w / H ** 3
        t = bar[at] * m[j] * KN / H ** 4 * np.divide(dw, r, out=np.zeros_like(r), where=r > 0)
        for a, i in ((0, 2), (1, 1), (2, 0)):
            grad[a, j] = (t * d[a][k[i]]).sum()
        grad[3, j] = -(bar[at] * m[j] * GK * KN / H ** 4 * (3 * w + q * dw)).sum()
    return rho, grad


@pytest.mark.parametrize("n,ng,h_lo,h_hi", [(1, 9, 0.1, 0.1), (33, 80, 0.1, 0.13), (40, 45, 1e-4, 0.25),
                                            (2500, 16, 0.01, 0.06), (5003, 8, 1e-3, 0.05),
                                            (4099, 10, 0.02, 0.09)])
def test_grid_density_and_adjoint(env, n, ng, h_lo, h_hi):
    torch, sim = env
    rng = np.random.default_rng(n + ng)
    pos = rng.uniform(0, 1, size=(n, 3))
    pos[0] = (np.array([0, ng // 2, ng - 1]) + 0.5) / ng  # on a grid point, at the box's edge
    h = np.exp(rng.uniform(np.log(h_lo), np.log(h_hi), size=n)).astype(np.float32)
    m = rng.uniform(0.5, 1.5, size=n).astype(np.float32)
    vel = rng.normal(size=(n, 3)).astype(np.float32)
    vel[0] = 0.0
    dt = 1e-5
    bar = rng.normal(size=ng ** 3)
    p = sim.Particles(n)
    for k, name in enumerate("xyz"):
        getattr(p, name).copy_(torch.as_tensor(pos[:, k].copy()))
        getattr(p, "v" + name).copy_(torch.as_tensor(vel[:, k].copy()))
    p.m.copy_(torch.as_tensor(m))
    p.h.copy_(torch.as_tensor(h))
    p.ti_drift.fill_(3)
    ctx = sim.Context(sim.Params(dt_min=dt), n)
    adj = sim.Adjoint(n)
    rho = ctx.grid_density(p, ng, 103).cpu().numpy()
    ctx.grid_density_bwd(p, ng, 103, torch.as_tensor(bar, device="cuda"), adj)
    x = pos + vel.astype(np.float64) * (100 * dt)
    want, grad = direct(x, m.astype(np.float64), h.astype(np.float64), bar, ng)
    # FP64 throughout: a support of N points sums N terms of either sign, a grid
    # point at most n; the offsets carry an absolute error of 2^-52 of the box,
    # magnified by 1 / H (and once more in the derivatives)
    points = 4.19 * (GK * h_hi * ng) ** 3 + n
    tol = 4 * 2.0 ** -52 * (points + 30 / (GK * h_lo))
    assert np.abs(rho - want).max() <= tol * np.abs(want).max()
    got = [getattr(adj, k).cpu().numpy() for k in ("x", "y", "z", "h")]
    for g, w in zip(got, grad):
        assert np.abs(g - w).max() <= tol * np.abs(w).max()
    for k, name in enumerate(("vx", "vy", "vz")):
        v = getattr(adj, name).cpu().numpy()
        assert np.allclose(v, got[k] * (100 * dt), rtol=1e-14, atol=0)
