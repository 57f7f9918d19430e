"""A cell build whose bounded waits give up (the checks build's planted stall:
one tile keeps its counts to itself): the call returns SPH_ERR_TIMEOUT, the
particles are still the same set, there are no cells, and the next build is the
one that an undisturbed context makes.  And builds where no thread-block cluster
can be placed.  Both in a child process that loads the checks build."""
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if __name__ != "__main__":
    pytestmark = pytest.mark.gpu
N, NC = 70001, 20  # 18 tiles of particles, several of leaves


def _state(sim, torch, seed):
    rng = np.random.default_rng(seed)
    p = sim.Particles(N)
    for name in "xyz":
        getattr(p, name).copy_(torch.as_tensor(rng.uniform(size=N)))
    p.m.copy_(torch.as_tensor(np.arange(N) + 1.0, dtype=torch.float32))  # who is who
    p.h.fill_(0.01)
    p.A.fill_(1.0)
    return p


def _run(stage, wait_limit):
    """One build that gives up, then one that does not; what both left."""
    import torch
    from paper_1807_01341_gb300 import _lib, sim
    out = {}
    ctx = sim.Context(sim.Params(n_cells_override=NC, leaf_max=4, wait_limit=wait_limit,
                                 test_build_stall=stage), N)
    p = _state(sim, torch, 5)
    try:
        ctx.build_cells(p)
        out["code"] = 0
    except _lib.SphError as e:
        out["code"] = e.code
    out["who_failed"] = p.m.cpu().numpy()
    out["x_failed"] = p.x.cpu().numpy()
    try:
        ctx.mark_active(p, 0)
        out["mark"] = 0
    except _lib.SphError as e:
        out["mark"] = e.code
    saved = sim.Particles(N)
    ctx.state_copy(p, saved, True)
    out["who_copied"] = saved.m.cpu().numpy()
    ctx.build_cells(p)
    out["who"], out["x"], out["perm"] = p.m.cpu().numpy(), p.x.cpu().numpy(), ctx.perm_tensor(N).cpu().numpy()
    out["info"] = ctx.grid_info()
    out["status"] = ctx.status()[0]
    ctx.close()
    return out


def _run_without_clusters():
    """Builds of sizes that a cluster sorts, with and without one."""
    import torch
    from paper_1807_01341_gb300 import sim
    out = []
    for n in (1, 4097, 16385, 40000, 65536):
        rng = np.random.default_rng(n)
        pos = rng.uniform(size=(n, 3))
        perms, launches, infos = [], [], []
        for stall in (0, 4):
            ctx = sim.Context(sim.Params(n_cells_override=20, test_build_stall=stall), n)
            p = sim.Particles(n)
            for k, name in enumerate("xyz"):
                getattr(p, name).copy_(torch.as_tensor(pos[:, k].copy()))
            p.m.fill_(1.0)
            p.h.fill_(0.01)
            before = ctx.counters()["kernel_launches"]
            ctx.build_cells(p)
            launches.append(ctx.counters()["kernel_launches"] - before)
            perms.append(ctx.perm_tensor(n).cpu().numpy())
            infos.append(ctx.grid_info())
            ctx.close()
        out.append(dict(pos=pos, perms=perms, launches=launches, infos=infos))
    return out


@pytest.fixture(scope="module")
def plain():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1807_01341_gb300 import build
    build.build()
    from paper_1807_01341_gb300 import _lib, sim
    return torch, _lib, sim


@pytest.mark.parametrize("stage,wait_limit", [(1, 1), (2, 1), (3, 1), (1, 5000), (2, 5000)])
def test_build_gives_up_and_recovers(plain, tmp_path, stage, wait_limit):
    torch, _lib, sim = plain
    path = str(tmp_path / "out.npy")
    env = dict(os.environ, SPH_GB300_CHECKS="1", PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, os.path.abspath(__file__), str(stage), str(wait_limit), path],
                       env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    got = np.load(path, allow_pickle=True).item()
    assert got["code"] == _lib.SPH_ERR_TIMEOUT
    assert got["mark"] == _lib.SPH_ERR_NOT_BUILT
    ctx = sim.Context(sim.Params(n_cells_override=NC, leaf_max=4), N)
    p = _state(sim, torch, 5)
    x = p.x.cpu().numpy()
    ctx.build_cells(p)
    # nothing lost and nobody changed places without its arrays
    assert np.array_equal(np.sort(got["who_failed"]), np.arange(N) + 1.0)
    assert np.array_equal(got["x_failed"], x[got["who_failed"].astype(np.int64) - 1])
    # copies to the input order, and the next build's permutation, are still
    # relative to the order before the first build
    assert np.array_equal(got["who_copied"], np.arange(N) + 1.0)
    assert np.array_equal(got["perm"], got["who"].astype(np.int64) - 1)
    # the next build: the same order and cells
    assert np.array_equal(got["who"], p.m.cpu().numpy())
    assert np.array_equal(got["x"], p.x.cpu().numpy())
    assert got["info"] == ctx.grid_info()
    assert got["status"] == 0
    ctx.close()


def test_build_without_clusters(plain, tmp_path):
    from test_gpu_build import keys_of
    path = str(tmp_path / "out.npy")
    env = dict(os.environ, SPH_GB300_CHECKS="1", PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, os.path.abspath(__file__), "4", "0", path], env=env,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    for got in np.load(path, allow_pickle=True):
        want = np.argsort(keys_of(got["pos"], 20)[1], kind="stable")
        for perm in got["perms"]:
            assert np.array_equal(perm, want)
        assert got["infos"][0] == got["infos"][1]
        # (43 bits of key: one launch where a cluster sorts, else six)
        assert got["launches"][1] - got["launches"][0] == 5


def test_short_wait_limit_leaves_builds_alone(plain):
    """wait_limit = 1: the waits of an undisturbed build are longer than that."""
    torch, _lib, sim = plain
    n = 1 << 20
    ctx = sim.Context(sim.Params(n_cells_override=40, wait_limit=1), n)
    p = sim.Particles(n)
    for name in "xyz":
        getattr(p, name).uniform_()
    p.m.fill_(1.0)
    p.h.fill_(0.01)
    for _ in range(5):
        ctx.build_cells(p)
    assert ctx.grid_info()[0] == 40
    ctx.close()


if __name__ == "__main__":
    sys.path.insert(0, ROOT)
    stage = int(sys.argv[1])
    res = _run_without_clusters() if stage == 4 else _run(stage, int(sys.argv[2]))
    np.save(sys.argv[3], res, allow_pickle=True)
