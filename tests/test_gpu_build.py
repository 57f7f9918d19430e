"""The cell build's order and leaf count at the edges of its tiles and of its
key arithmetic, against the definition in numpy: cell and Morton coordinate by
the FP64 divisions, a stable sort, and the octree split node by node."""
import numpy as np
import pytest

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


def keys_of(pos, nc, box=1.0):
    w = box / nc
    x = np.where(pos < 0, pos + box, pos)
    x = np.where(x >= box, x - box, x)
    c = np.clip(np.floor(x / w), 0, nc - 1)
    t = (x - c * w) / w * 1024.0
    q = np.clip(np.floor(t), 0, 1023).astype(np.uint64)
    c = c.astype(np.uint64)
    key = (c[:, 0] * np.uint64(nc) + c[:, 1]) * np.uint64(nc) + c[:, 2]
    key = key << np.uint64(30)
    for b in range(10):
        for a in range(3):
            key |= ((q[:, a] >> np.uint64(b)) & np.uint64(1)) << np.uint64(3 * b + 2 - a)
    return x, key


def count_leaves(keys, leaf_max):
    """Leaves of sorted keys, by the recursive definition of the split."""
    def split(a, b, level):
        if level == 10:
            return -(-(b - a) // leaf_max)
        d = (keys[a:b] >> np.uint64(3 * (9 - level))) & np.uint64(7)
        n, run = 0, 0
        for k in range(8):
            lo, hi = a + np.searchsorted(d, k), a + np.searchsorted(d, k, side="right")
            c = hi - lo
            if c == 0:
                continue
            if c > leaf_max:
                n, run = n + split(lo, hi, level + 1), 0
            elif run and run + c <= leaf_max:
                run += c
            else:
                n, run = n + 1, c
        return n
    cells = keys >> np.uint64(30)
    edges = np.flatnonzero(np.r_[True, cells[1:] != cells[:-1], True])
    return sum(1 if b - a <= leaf_max else split(a, b, 0) for a, b in zip(edges[:-1], edges[1:]))


def positions(kind, n, nc, rng):
    pos = rng.uniform(0, 1, size=(n, 3))
    if kind == "edges":  # whole Morton steps, their neighbours in FP64, and the box's ends
        pos = rng.integers(0, nc * 1024 + 1, size=(n, 3)) / (nc * 1024.0)
        pos = np.nextafter(pos, rng.choice([-1.0, 0.5, 2.0], size=(n, 3)))
        pos = np.where(rng.uniform(size=(n, 3)) < 0.3, np.round(pos * nc) * (1.0 / nc), pos)
        pos[rng.integers(0, n, size=n // 8), rng.integers(0, 3, size=n // 8)] += 1.0
        pos[rng.integers(0, n, size=n // 8), rng.integers(0, 3, size=n // 8)] -= 1.0
    if kind == "clumps":  # equal positions, and clumps below a Morton step
        pos[n // 3:] = pos[rng.integers(0, min(n, 5), size=n - n // 3)]
        pos[n // 2:] += rng.uniform(0, 1e-4 / nc, size=(n - n // 2, 3))
        pos[n - n // 5:] = pos[0] + rng.normal(size=(n // 5, 3)) * 0.01
        pos -= np.floor(pos)
    return pos


@pytest.mark.parametrize("n,nc,leaf_max", [(1, 3, 8), (31, 3, 1), (4095, 5, 8), (4096, 3, 32),
                                           (4097, 40, 16), (65537, 7, 8), (70001, 255, 3)])
@pytest.mark.parametrize("kind", ["uniform", "edges", "clumps"])
def test_order_and_leaves(env, n, nc, leaf_max, kind):
    torch, sim = env
    rng = np.random.default_rng(n + nc)
    pos = positions(kind, n, nc, rng)
    ctx = sim.Context(sim.Params(n_cells_override=nc, leaf_max=leaf_max), n)
    p = sim.Particles(n)
    for k, name in enumerate("xyz"):
        getattr(p, name).copy_(torch.as_tensor(pos[:, k].copy()))
    for k, t in enumerate(p.arrays().values()):  # every array travels with its particle
        if t.data_ptr() not in (p.x.data_ptr(), p.y.data_ptr(), p.z.data_ptr()):
            t.copy_((torch.arange(n) * 7 + k) % 50 + 1)
    before = {k: t.cpu().numpy().copy() for k, t in p.arrays().items()}
    ctx.build_cells(p)
    perm = ctx.perm_tensor(n).cpu().numpy()
    x, key = keys_of(pos, nc)
    assert np.array_equal(perm, np.argsort(key, kind="stable"))
    assert ctx.grid_info() == (nc, count_leaves(key[perm], leaf_max))
    before.update(x=x[:, 0], y=x[:, 1], z=x[:, 2])
    for name, t in p.arrays().items():
        if name in ("P", "c"):  # (the build's refresh computes them from the other arrays)
            continue
        want = np.zeros(n, np.uint8) if name == "active" else before[name][perm]
        assert np.array_equal(t.cpu().numpy(), want), name
    counts = np.bincount(before["bin"], minlength=64)
    assert ctx.bin_counts() == counts.tolist()
    # a second build composes the order: it stays relative to the first input
    # (a position more than one box length outside is wrapped once more)
    ctx.build_cells(p)
    again = perm[np.argsort(keys_of(x[perm], nc)[1], kind="stable")]
    assert np.array_equal(ctx.perm_tensor(n).cpu().numpy(), again)


@pytest.mark.parametrize("n,nc", [(8191, 8), (8193, 64), (16384, 20), (16384, 65), (16385, 11),
                                  (32768, 64), (32769, 30), (49152, 40), (49153, 40), (65535, 64),
                                  (65536, 16), (65536, 65)])
def test_order_of_one_cluster(env, n, nc):
    """The sizes up to 65,536 and keys up to 48 bits (64 cells per axis) that
    one cluster sorts: the edges of its instances, and both ends of the rule."""
    torch, sim = env
    rng = np.random.default_rng(n * 100 + nc)
    pos = positions("uniform" if n % 2 else "clumps", n, nc, rng)
    pos[rng.integers(0, n, size=n // 16)] = np.nextafter(1.0, 0.0)  # the largest key, many times
    ctx = sim.Context(sim.Params(n_cells_override=nc, leaf_max=16), n)
    p = sim.Particles(n)
    p.m.fill_(1.0)
    p.h.fill_(0.01)
    for k, name in enumerate("xyz"):
        getattr(p, name).copy_(torch.as_tensor(pos[:, k].copy()))
    for _ in range(2):  # the second one starts from the sorted order
        ctx.build_cells(p)
        key = keys_of(pos, nc)[1]
        perm = ctx.perm_tensor(n).cpu().numpy()
        assert np.array_equal(perm, np.argsort(key, kind="stable"))
        assert ctx.grid_info() == (nc, count_leaves(key[perm], 16))
