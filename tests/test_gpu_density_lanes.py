"""Several lanes per particle whose lists fill up: further passes over the
candidates, in which some lanes of a particle have nothing left to list.  h and
rho against the FP64 oracle, at the tolerance of the other density tests."""
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
    import oracle
    oracle.build()
    from paper_1807_01341_gb300 import sim
    return torch, sim, oracle


@pytest.mark.parametrize("lanes", [2, 4, 8, 16, 32])
@pytest.mark.parametrize("cap,depth", [(32, 1), (33, 3), (100, 1)])
def test_against_the_oracle(env, lanes, cap, depth):
    torch, sim, oracle = env
    ic = sph_ics.lattice(17, 0.1, seed=5)
    ic["h0"] = ic["h0"] * np.random.default_rng(lanes).uniform(0.5, 2.3, ic["pos"].shape[0])
    ctx, p = gpu_setup(ic, sim.Params(list_cap=cap, threads_per_particle=lanes, cell_margin=1.2,
                                      staging_depth=depth))
    ctx.mark_active(p, 0)
    ctx.kick_drift(p, 0)
    ctx.density_active(p, 1)
    assert ctx.status()[0] == 0
    assert ctx.counters()["list_overflows"] > 0 or lanes * cap > 500
    s = sorted_inputs(ic, ctx.perm_tensor(p.n).cpu().numpy())
    ref = oracle.density(s["pos"], s["m"].astype(np.float32).astype(np.float64),
                         s["h0"].astype(np.float32).astype(np.float64))
    assert np.abs(p.h.cpu().numpy() / ref["h"] - 1).max() < 1e-5
    assert np.abs(p.rho.cpu().numpy() / ref["rho"] - 1).max() < 1e-5
