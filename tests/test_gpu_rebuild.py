"""What a cell build leaves behind it: the work queues of the structure before
it, the composed permutation, and a build that is refused or gives up."""
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


def host(p):
    return {k: t.cpu().numpy().copy() for k, t in p.arrays().items()}


@pytest.mark.parametrize("list_cap", [32, 512])
def test_no_queue_survives_a_build(env, list_cap):
    """Active set, density (with particles over their list, and heavy groups),
    then a build: the passes find no active particle until the next marking."""
    torch, sim = env
    ic = sph_ics.clumpy_lattice(17, 3, 500, seed=7)
    n = ic["pos"].shape[0]
    ctx = sim.Context(sim.Params(list_cap=list_cap, leaf_max=16,
                                 heavy_factor=0.5), n)
    p = sim.Particles.from_ics(ic)
    ctx.resume(p, 0, True)
    ctx.build_cells(p)
    ctx.mark_active(p, 0)
    ctx.density_active(p, 1)
    assert ctx.status()[0] == 0
    if list_cap == 32:
        assert ctx.counters()["list_overflows"] > 0
    p.h.mul_(0.9)  # another grid, fewer groups and chunks than indices in the old queues
    ctx.build_cells(p)
    before = host(p)
    ctx.kick_drift(p, 0)
    ctx.density_active(p, 0)
    ctx.force_active(p)
    ctx.kick_drift(p, 1)
    ctx.timestep_bins(p)
    ctx.kick_drift(p, 2)
    after = host(p)
    for k in before:
        assert np.array_equal(before[k], after[k], equal_nan=True), k
    assert ctx.status()[0] == 0
    ctx.mark_active(p, 0)  # and the next marking starts from a clean slate
    ctx.density_active(p, 0)
    assert p.active.all()
    assert np.array_equal(p.rho.cpu().numpy() > 0, np.ones(n, bool))


@pytest.mark.parametrize("sizes", [(0, 3000), (1000, 3000), (3000, 1000, 2500)])
def test_builds_of_growing_sets(env, sizes):
    """Particles that an earlier build of the context did not hold start the
    composed permutation at their own place, and every array keeps its bytes."""
    torch, sim = env
    rng = np.random.default_rng(11)
    big = max(sizes)
    # (memory that was used before: a new allocation is not zero)
    junk = torch.full((1 << 28,), -1, dtype=torch.int8, device="cuda")
    del junk
    torch.cuda.empty_cache()
    ctx = sim.Context(sim.Params(n_cells_override=7), big)
    perm = np.arange(0)
    for n in sizes:
        p = sim.Particles(n)
        for name in "xyz":
            getattr(p, name).copy_(torch.as_tensor(rng.uniform(size=n)))
        p.m.fill_(1.0)
        p.h.copy_(torch.as_tensor(rng.uniform(0.01, 0.02, size=n), dtype=torch.float32))
        p.bin.copy_(torch.as_tensor(rng.integers(0, 50, size=n), dtype=torch.int8))
        before = host(p)
        ctx.build_cells(p)
        if n == 0:
            continue
        now = host(p)
        at = np.argsort(before["x"])[np.argsort(np.argsort(now["x"]))]  # who stands where
        for name in ("x", "h", "bin"):
            assert np.array_equal(now[name], before[name][at]), name
        assert ctx.bin_counts() == np.bincount(before["bin"], minlength=64).tolist()
        old = np.r_[perm[:n], np.arange(min(perm.size, n), n)]
        perm = old[at]
        assert np.array_equal(ctx.perm_tensor(n).cpu().numpy(), perm)


@pytest.mark.parametrize("finer", [True, False])
def test_refused_build(env, finer):
    """A build refused for a position that is no number: the cells before it
    stay in use, or, where the new grid needed larger arrays, there are none
    until a build succeeds; the particles and their permutation stay."""
    torch, sim = env
    from paper_1807_01341_gb300 import _lib
    n = 4000
    rng = np.random.default_rng(2)
    ctx = sim.Context(sim.Params(), n)
    p = sim.Particles(n)
    for name in "xyz":
        getattr(p, name).copy_(torch.as_tensor(rng.uniform(size=n)))
    p.m.copy_(torch.arange(n) + 1.0)
    p.h.fill_(0.06)
    p.A.fill_(1.0)
    ctx.build_cells(p)
    info, perm = ctx.grid_info(), ctx.perm_tensor(n).cpu().numpy()
    x0 = float(p.x[0])
    p.x[0] = float("nan")
    p.h.fill_(0.004 if finer else 0.09)
    who = p.m.cpu().numpy()
    with pytest.raises(_lib.SphError) as e:
        ctx.build_cells(p)
    assert e.value.code == _lib.SPH_ERR_ARG
    assert np.array_equal(p.m.cpu().numpy(), who)
    assert np.array_equal(ctx.perm_tensor(n).cpu().numpy(), perm)
    p.x[0] = x0
    p.h.fill_(0.06)
    if finer:
        with pytest.raises(_lib.SphError) as e:
            ctx.mark_active(p, 0)
        assert e.value.code == _lib.SPH_ERR_NOT_BUILT
    else:
        assert ctx.grid_info() == info
        ctx.mark_active(p, 0)
        ctx.density_active(p, 1)
        assert ctx.status()[0] == 0 and p.active.all()
    saved = sim.Particles(n)
    ctx.state_copy(p, saved, True)
    assert np.array_equal(saved.m.cpu().numpy(), np.arange(n) + 1.0)
    ctx.resume(p, 0, True)
    ctx.step(p, 1)
    assert ctx.counters()["steps"] == 1


@pytest.mark.parametrize("n", [1, 4097, 1 << 20, (1 << 20) + 5])
@pytest.mark.parametrize("optional", [True, False])
def test_copy_to_the_input_order(env, n, optional):
    """Every array back in the order before the build, byte for byte."""
    torch, sim = env
    ctx = sim.Context(sim.Params(n_cells_override=30), n)
    p = sim.Particles(n, with_counts=optional, with_gradients=optional)
    g = torch.Generator(device="cuda").manual_seed(n)
    p.storage.copy_(torch.randint(0, 256, p.storage.shape, generator=g, device="cuda",
                                  dtype=torch.uint8))
    for name in "xyz":
        getattr(p, name).copy_(torch.rand(n, generator=g, device="cuda", dtype=torch.float64))
    p.h.fill_(0.01)
    p.m.fill_(1.0)
    p.bin.remainder_(60)
    p.rho.fill_(-1.0)  # (the build's refresh computes P and c where rho > 0)
    before = host(p)
    ctx.build_cells(p)
    out = sim.Particles(n, with_counts=optional)
    out.storage.fill_(7)
    ctx.state_copy(p, out, True)
    after = host(out)
    for name, a in before.items():
        if name != "active":
            assert np.array_equal(a.view(np.uint8), after[name].view(np.uint8)), name
    assert not after["active"].any()
    if not optional:
        assert (after["curl_v"].view(np.uint8) == 7).all()  # absent in one of the two: left alone


def test_copy_of_another_number_of_particles(env):
    """After builds of 3000 and then 1000 particles the permutation's indices
    reach 2999: a copy into 1000 places is refused, and so is one of more
    particles than it covers; a restart makes it fit again."""
    torch, sim = env
    from paper_1807_01341_gb300 import _lib
    ctx = sim.Context(sim.Params(n_cells_override=5), 3000)
    states = {}
    for n in (3000, 1000):
        p = states[n] = sim.Particles(n)
        for name in "xyz":
            getattr(p, name).uniform_()
        p.m.copy_(torch.arange(n) + 1.0)
        p.h.fill_(0.01)
        ctx.build_cells(p)
    for n in (1000, 3000):
        out = sim.Particles(n)
        with pytest.raises(_lib.SphError) as e:
            ctx.state_copy(states[n], out, True)
        assert e.value.code == _lib.SPH_ERR_ARG
        assert not out.storage.any()
    p = states[1000]
    who = p.m.cpu().numpy()
    ctx.resume(p, 0, True)
    ctx.build_cells(p)
    ctx.state_copy(p, out := sim.Particles(1000), True)
    assert np.array_equal(out.m.cpu().numpy(), who)
