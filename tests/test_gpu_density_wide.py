"""Many particles whose candidates outgrow their neighbour lists (a crude first
guess of h, or a short list): the density pass takes them a particle per lane
and the state does not depend on it, bit for bit; h and rho agree with the
oracle."""
import numpy as np
import pytest

import sph_ics
from _gpu_helpers import gpu_setup, sorted_inputs

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


def make(kind, masses):
    if kind == "wide":  # more than 8 particles per warp of the density grid, all over
        ic = sph_ics.lattice(31, 0.1, seed=5)
        ic["h0"] = ic["h0"] * 2.3
    elif kind == "mixed":  # some lanes of most warps
        ic = sph_ics.lattice(40, 0.1, seed=6)
        ic["h0"] = ic["h0"] * np.where(np.random.default_rng(1).uniform(size=64000) < 0.5, 2.3, 1.0)
    else:
        ic = sph_ics.clumpy_lattice(34, 6, 700, seed=7)
    if masses == "random":
        ic["m"] = ic["m"] * np.random.default_rng(3).uniform(0.5, 1.5, ic["m"].shape[0])
    return ic


@pytest.mark.parametrize("masses", ["equal", "random"])
@pytest.mark.parametrize("kind", ["wide", "mixed", "clumpy"])
def test_independent_of_list_capacity(env, kind, masses):
    torch, sim = env
    ic = make(kind, masses)
    n = ic["pos"].shape[0]
    got = {}
    for cap, form, depth in ((4096, 1, 1), (400, 1, 1), (32, 1, 1), (32, 0, 3)):
        ctx = sim.Context(sim.Params(list_cap=cap, dt_min=2.0 ** -26, leaf_max=16, cell_margin=1.2,
                                     staging_depth=depth), n)
        p = sim.Particles.from_ics(ic)
        ctx.resume(p, 0, True)
        for _ in range(2):
            ctx.step(p, form)
        got[cap, form] = {k: t.cpu().numpy() for k, t in p.arrays().items()}
        assert (ctx.counters()["list_overflows"] > (n // 2 if cap == 32 else 0)) == (cap < 4096)
        ctx.close()
    for key, state in got.items():
        for name, a in got[4096, 1].items():
            assert np.array_equal(a, state[name]), (key, name)


@pytest.mark.parametrize("masses", ["equal", "random"])
def test_against_the_oracle(env, masses):
    torch, sim = env
    import oracle
    oracle.build()
    ic = make("wide", masses)
    ctx, p = gpu_setup(ic, sim.Params(list_cap=32, cell_margin=1.2))
    ctx.mark_active(p, 0)
    ctx.kick_drift(p, 0)
    ctx.density_active(p, 1)
    n = p.n
    assert ctx.status()[0] == 0 and ctx.counters()["list_overflows"] == n
    s = sorted_inputs(ic, ctx.perm_tensor(n).cpu().numpy())
    ref = oracle.density(s["pos"], s["m"].astype(np.float32).astype(np.float64),
                         s["h0"].astype(np.float32).astype(np.float64))
    assert np.abs(p.h.cpu().numpy() / ref["h"] - 1).max() < 1e-5
    assert np.abs(p.rho.cpu().numpy() / ref["rho"] - 1).max() < 1e-5
    # the counters are those of a run whose lists hold every candidate
    got = ctx.counters()
    ctx2, p2 = gpu_setup(ic, sim.Params(list_cap=4096, cell_margin=1.2))
    ctx2.mark_active(p2, 0)
    ctx2.kick_drift(p2, 0)
    ctx2.density_active(p2, 1)
    want = ctx2.counters()
    assert want["list_overflows"] == 0
    for k in ("pairs_density", "iters_density"):
        assert got[k] == want[k], k
    assert np.array_equal(p.ngb_density.cpu().numpy(), p2.ngb_density.cpu().numpy())
