"""The cell build past the first windows of its look-backs (32 tiles of 4,096):
the exact order and leaf count, and every particle reached through the chunks
and work groups."""
import numpy as np
import pytest

from test_gpu_build import count_leaves, keys_of, positions

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


@pytest.mark.parametrize("n,nc,leaf_max,kind", [(131072, 20, 8, "uniform"), (131073, 20, 8, "uniform"),
                                                (200003, 9, 16, "clumps"), (1000003, 60, 8, "uniform"),
                                                (1000003, 40, 16, "clumps"), (1300000, 70, 1, "uniform")])
def test_order_and_leaves(env, n, nc, leaf_max, kind):
    torch, sim = env
    pos = positions(kind, n, nc, np.random.default_rng(n + nc))
    ctx = sim.Context(sim.Params(n_cells_override=nc, leaf_max=leaf_max), n)
    p = sim.Particles(n)
    for k, name in enumerate("xyz"):
        getattr(p, name).copy_(torch.as_tensor(pos[:, k].copy()))
    p.m.copy_(torch.arange(n) + 1.0)
    p.h.fill_(0.1 / nc)
    ctx.build_cells(p)
    key = keys_of(pos, nc)[1]
    perm = np.argsort(key, kind="stable")
    assert np.array_equal(ctx.perm_tensor(n).cpu().numpy(), perm)
    assert np.array_equal(p.m.cpu().numpy(), (perm + 1).astype(np.float32))
    if kind == "uniform" and leaf_max > 1:
        assert ctx.grid_info() == (nc, count_leaves(key[perm], leaf_max))
    # every particle is marked, and drifted through its chunk
    p.vx.fill_(1.0)
    ctx.mark_active(p, 1 << 10)
    assert p.active.all()
    ctx.kick_drift(p, 0)
    assert (p.ti_drift == 1 << 10).all()


def test_every_particle_is_in_a_work_group(env):
    """The density pass reaches every particle of a set of 40 tiles."""
    torch, sim = env
    n = 160001
    side = 55
    rng = np.random.default_rng(4)
    c = (np.arange(side) + 0.5) / side
    pos = np.stack(np.meshgrid(c, c, c, indexing="ij"), -1).reshape(-1, 3)[:n]
    pos = np.r_[pos, pos[rng.integers(0, len(pos), size=n - len(pos))] + 0.2 / side][:n]
    pos += rng.uniform(-0.1, 0.1, size=pos.shape) / side
    pos -= np.floor(pos)
    ctx = sim.Context(sim.Params(), n)
    p = sim.Particles(n)
    for k, name in enumerate("xyz"):
        getattr(p, name).copy_(torch.as_tensor(pos[:, k].copy()))
    p.m.fill_(1.0 / n)
    p.A.fill_(1.0)
    p.h.fill_(1.2348 / side)
    ctx.build_cells(p)
    ctx.mark_active(p, 0)
    ctx.kick_drift(p, 0)
    ctx.density_active(p, 1)
    ctx.force_active(p)
    assert ctx.status()[0] == 0
    assert (p.rho > 0).all() and (p.vsig > 0).all()
    assert (p.ngb_density > 20).all()
