"""A step that halts because a support outgrew its cell is redone on wider cells
whatever other errors were recorded before that one: particles whose h did not
converge do not stop it, in either order."""
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
    from paper_1807_01341_gb300 import _lib, sim
    return torch, _lib, sim


@pytest.mark.parametrize("list_cap", [512, 64])
def test_redone_beside_unconverged_particles(env, list_cap):
    torch, _lib, sim = env
    ic = sph_ics.lattice(20, 0.1, seed=111)
    g = np.random.default_rng(111)
    n = ic["pos"].shape[0]
    ic["pos"] = (0.95 + 0.2 * g.normal(size=(n, 3))) % 1.0
    ic["h0"] = ic["h0"] * 0.5
    outcomes = set()
    for _ in range(8):
        ctx = sim.Context(sim.Params(dt_min=2.0 ** -26, bin_cap=4, leaf_max=3, cell_margin=3.0,
                                     h_max_iter=4, list_cap=list_cap), n)
        p = sim.Particles.from_ics(ic)
        ctx.resume(p, 0, True)
        ctx.step(p, 1)
        c = ctx.counters()
        outcomes.add((ctx.status()[0], c["steps"], c["redone_steps"] > 0, c["pairs_density"],
                      p.h.cpu().numpy().tobytes()))
        ctx.close()
    assert len(outcomes) == 1
    status, steps, redone = next(iter(outcomes))[:3]
    assert (status, steps, redone) == (_lib.SPH_ERR_H_NOCONV, 1, True)
