"""Grid density and its adjoint where a support holds no point or is no number."""
import numpy as np
import pytest

from test_gpu_grid import direct

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1807_01341_gb300 import build
    build.build()
    from paper_1807_01341_gb300 import sim
    return torch, sim


def state(sim, torch, pos, m, h):
    p = sim.Particles(len(m))
    for k, name in enumerate("xyz"):
        getattr(p, name).copy_(torch.as_tensor(pos[:, k].copy()))
    p.m.copy_(torch.as_tensor(m))
    p.h.copy_(torch.as_tensor(h))
    return p


@pytest.mark.parametrize("n,ng", [(40, 9), (3000, 8)])
@pytest.mark.parametrize("odd", [0.0, -0.01, np.nan, 1e-30])
def test_supports_without_a_point(env, n, ng, odd):
    """Particles whose h is zero (one of them on a grid point), negative, not a
    number or tiny leave the grid and every adjoint as they are."""
    torch, sim = env
    rng = np.random.default_rng(n)
    pos = rng.uniform(size=(n, 3))
    m = rng.uniform(0.5, 1.5, size=n).astype(np.float32)
    h = rng.uniform(0.02, 0.09, size=n).astype(np.float32)
    off = np.arange(n) % 3 == 0
    h[off] = odd
    if odd <= 0.0:
        pos[0] = 0.5 / ng
    bar = rng.normal(size=ng ** 3)
    p = state(sim, torch, pos, m, h)
    ctx = sim.Context(sim.Params(), n)
    adj = sim.Adjoint(n)
    for k, name in enumerate(("x", "y", "z", "h")):
        getattr(adj, name).fill_(k + 1.0)
    rho = ctx.grid_density(p, ng, 0).cpu().numpy()
    ctx.grid_density_bwd(p, ng, 0, torch.as_tensor(bar, device="cuda"), adj)
    want, grad = direct(pos[~off], m[~off].astype(float), h[~off].astype(float), bar, ng)
    assert np.allclose(rho, want, rtol=1e-12, atol=1e-12 * want.max())
    for k, name in enumerate(("x", "y", "z", "h")):
        got = getattr(adj, name).cpu().numpy()
        assert np.array_equal(got[off], np.full(off.sum(), k + 1.0)), name
        assert np.allclose(got[~off] - (k + 1.0), grad[k], rtol=1e-9, atol=1e-9 * np.abs(grad[k]).max())


@pytest.mark.parametrize("n,ng,h_lo,h_hi", [(4099, 8, 0.01, 0.03), (2048, 5, 0.02, 0.05),
                                            (3001, 16, 0.005, 0.02)])
def test_boxes_of_a_point_or_none(env, n, ng, h_lo, h_hi):
    """Supports narrower than the grid's spacing, most of which miss every
    point: a few lanes of a warp with a point each."""
    torch, sim = env
    rng = np.random.default_rng(ng)
    pos = rng.uniform(size=(n, 3))
    pos[::500] = 0.5 / ng + rng.integers(0, ng, size=(len(pos[::500]), 3)) / ng
    m = rng.uniform(0.5, 1.5, size=n).astype(np.float32)
    h = rng.uniform(h_lo, h_hi, size=n).astype(np.float32)
    bar = rng.normal(size=ng ** 3)
    p = state(sim, torch, pos, m, h)
    ctx = sim.Context(sim.Params(), n)
    adj = sim.Adjoint(n)
    rho = ctx.grid_density(p, ng, 0).cpu().numpy()
    ctx.grid_density_bwd(p, ng, 0, torch.as_tensor(bar, device="cuda"), adj)
    want, grad = direct(pos, m.astype(float), h.astype(float), bar, ng)
    # sums of at most n positive terms; an offset's error, 2^-52 of the box, grows
    # by 1 / H where the kernel falls off
    tol = 4 * 2.0 ** -52 * (n + 30 / (1.825742 * h_lo))
    assert np.abs(rho - want).max() <= tol * want.max()
    for name, g in zip(("x", "y", "z", "h"), grad):
        assert np.abs(getattr(adj, name).cpu().numpy() - g).max() <= tol * np.abs(g).max(), name


def bounds(x, m, h, bar, ng):
    """Direct sums as in `direct`, each with the sum of what its terms may be off:
    a relative error of 16 roundings and one for each term added, and the
    offsets' absolute error of 2^-52 of the box through the kernel's slope."""
    eps = 2.0 ** -52
    n = len(m)
    rho, drho, grad, dgrad = np.zeros(ng ** 3), np.zeros(ng ** 3), np.zeros((4, n)), np.zeros((4, n))
    c = (np.arange(ng) + 0.5) / ng
    for j in range(n):
        H = 1.825742 * h[j]
        d = [v - np.round(v) for v in (x[j, a] - c for a in range(3))]
        r2 = d[2][:, None, None] ** 2 + d[1][None, :, None] ** 2 + d[0][None, None, :] ** 2
        k = np.nonzero(r2 < H * H * (1 + 1e-12))
        r = np.sqrt(r2[k])
        q = np.minimum(r / H, 1.0)
        w = np.where(q < 0.5, 1 - 6 * q ** 2 + 6 * q ** 3, 2 * (1 - q) ** 3)
        wq = np.where(q < 0.5, -12 + 18 * q, -6 * (1 - q) ** 2 / np.maximum(q, 0.5))  # w' / q
        w2 = np.where(q < 0.5, np.abs(-12 + 36 * q), 12 * (1 - q))
        at = k[2] + ng * (k[1] + ng * k[0])
        C = m[j] * 2.5464790894703255 / H ** 3
        off = 4 * eps / H  # of q
        rho[at] += C * w
        drho[at] += C * (eps * (16 + n) * w + off * np.abs(wq * q) + off ** 2 * 12)
        t = bar[at] * C / H
        big = np.abs(t) * (eps * (16 + len(q)) * np.abs(wq) * q + off * (np.abs(wq) + w2 + 12 * off))
        for a, i in ((0, 2), (1, 1), (2, 0)):
            grad[a, j] = (t * wq * d[a][k[i]] / H).sum()
            dgrad[a, j] = big.sum()
        t = bar[at] * C * 1.825742 / H
        wh = 3 * w + q * q * wq
        grad[3, j] = -(t * wh).sum()
        dgrad[3, j] = (np.abs(t) * (eps * (16 + len(q)) * (3 * w + q * q * np.abs(wq)) +
                                    off * (4 * np.abs(wq * q) + q * w2 + 48 * off))).sum()
    return rho, drho, grad, dgrad


@pytest.mark.parametrize("n,ng,h_lo,h_hi", [(33, 80, 0.1, 0.13), (40, 45, 1e-4, 0.25),
                                            (700, 24, 1e-3, 0.2)])
def test_each_point_and_particle(env, n, ng, h_lo, h_hi):
    """Every grid point and every particle against the bound of its own terms,
    narrow supports beside wide ones of many tiles."""
    torch, sim = env
    rng = np.random.default_rng(n * ng)
    pos = rng.uniform(size=(n, 3))
    h = np.exp(rng.uniform(np.log(h_lo), np.log(h_hi), size=n)).astype(np.float32)
    m = rng.uniform(0.5, 1.5, size=n).astype(np.float32)
    bar = rng.normal(size=ng ** 3)
    p = state(sim, torch, pos, m, h)
    ctx = sim.Context(sim.Params(), n)
    adj = sim.Adjoint(n)
    rho = ctx.grid_density(p, ng, 0).cpu().numpy()
    ctx.grid_density_bwd(p, ng, 0, torch.as_tensor(bar, device="cuda"), adj)
    want, drho, grad, dgrad = bounds(pos, m.astype(float), h.astype(float), bar, ng)
    assert (np.abs(rho - want) <= drho).all()
    for name, g, dg in zip(("x", "y", "z", "h"), grad, dgrad):
        assert (np.abs(getattr(adj, name).cpu().numpy() - g) <= dg).all(), name
