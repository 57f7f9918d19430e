"""The passes of a step inside a caller's own CUDA graph: the device's time and
state after its replays are what every later call sees."""
import numpy as np
import pytest

import sph_ics

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


def passes(ctx, p):
    ctx.mark_active(p, -1)
    ctx.kick_drift(p, 0)
    ctx.density_active(p, 0)
    ctx.force_active(p)
    ctx.kick_drift(p, 1)
    ctx.timestep_bins(p)
    ctx.kick_drift(p, 2)


@pytest.mark.parametrize("list_cap", [512, 32])
def test_time_after_replays(env, list_cap):
    torch, sim = env
    ic = sph_ics.clumpy_lattice(12, 2, 150, seed=3)
    n = ic["pos"].shape[0]
    runs = []
    for captured in (False, True):
        ctx = sim.Context(sim.Params(dt_min=2.0 ** -22, bin_cap=8, list_cap=list_cap), n)
        p = sim.Particles.from_ics(ic)
        ctx.resume(p, 0, True)
        ctx.step(p, 1)
        if captured:
            assert ctx.get_time() == ctx.synced_time()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                passes(ctx, p)
            ctx.step(p, 1)  # (reads the device's time on the host)
            for _ in range(3):
                g.replay()
            torch.cuda.synchronize()
        else:
            ctx.step(p, 1)
            for _ in range(3):
                passes(ctx, p)
        runs.append((ctx.get_time(), ctx.status()[0], {k: t.cpu().numpy() for k, t in p.arrays().items()}))
    (ta, sa, a), (tb, sb, b) = runs
    assert ta == tb and sa == sb == 0
    for k in a:
        assert np.array_equal(a[k], b[k]), k
