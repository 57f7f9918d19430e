"""The work that a user of this library has it do, as measurable cases.

A program holds a particle state on the device and a context.  It starts (or
restarts) the state from a checkpoint, which rebuilds the cells, then takes
kick-drift-kick steps, either through the whole-step calls or pass by pass;
it differentiates a run; or it samples a state's density on a grid.  Each case
does that from a checkpoint held on the device, so that a pass can be repeated.

Kinds of case:
  passes    restart, then the calls of one step one by one (cells, active set,
            drift, density, force, kicks, bins), the state in the caller's order
  first     restart, then whole steps from the initial conditions with every
            particle active in the first one
  build     restart and the cell build alone
  run       restart, then a run of whole steps of which only the first has every
            particle active (the multiple-time-step workload)
  gradient  forward run and reverse pass of the grid-density loss (autograd)
  grid      grid density of a state and its adjoint

The particle sets are those of the repository's workloads (jittered lattices,
Sedov blasts, Plummer spheres in a uniform background, clumpy and
Zel'dovich-displaced lattices), drawn here on the GPU.
"""
import math

import torch

from paper_1807_01341_gb300 import _lib, adjoint, sim

ETA, GAMMA, GK, KN = 1.2348, 5.0 / 3.0, 1.825742, 2.5464790894703255
CFL, ALPHA = 0.1, 0.8
STATE_BYTES = 110   # one particle's state, without the optional arrays
NGB = 48            # neighbours of a particle at eta = 1.2348


def listed():
    return [
        # the smallest workload: 4,096 particles on one time bin, the calls one
        # by one with neighbour counts; latency and launches count
        dict(name="passes_4k", kind="passes", ics="lattice", nside=16, masses="equal", leaf_max=8,
             cell_margin=2.0, bin_cap=0, dt_min_log2=-13, steps=1, variants=False),
        # unequal masses (the general density loop) on an odd lattice
        dict(name="first_39k_masses", kind="first", ics="lattice", nside=34, masses="random",
             leaf_max=8, cell_margin=2.0, bin_cap=12, dt_min_log2=-24, steps=1, variants=False),
        # the 262,144-particle Sedov blast, bins up to 2^10
        dict(name="sedov_262k_run", kind="run", ics="sedov", nside=64, masses="equal", leaf_max=16,
             cell_margin=2.0, bin_cap=10, dt_min_log2=-24, steps=16, variants=False),
        # a blast with the Balsara switch, the prediction of inactive particles
        # and the time-step limiter switched on, as a production run has them
        dict(name="options_111k_run", kind="run", ics="sedov", nside=48, masses="equal", leaf_max=8,
             cell_margin=2.0, bin_cap=10, dt_min_log2=-24, steps=8, variants=True),
        # a mid-size clustered set, ragged sizes: mostly steps with few active
        # particles, where latency counts
        dict(name="clustered_302k_run", kind="run", ics="clustered", n_background=150001,
             n_spheres=37, per_sphere=4099, masses="equal", leaf_max=16, cell_margin=2.0,
             bin_cap=20, dt_min_log2=-28, steps=32, variants=False),
        # the benchmark's set: a cell build of 2,097,152 clustered particles
        dict(name="build_2m", kind="build", ics="clustered", n_background=1 << 20, n_spheres=64,
             per_sphere=1 << 14, masses="equal", leaf_max=16, cell_margin=2.0, bin_cap=20,
             dt_min_log2=-28, steps=0, variants=False),
        # the benchmark's workload: 20 steps of the same set
        dict(name="clustered_2m_run", kind="run", ics="clustered", n_background=1 << 20,
             n_spheres=64, per_sphere=1 << 14, masses="equal", leaf_max=16, cell_margin=2.0,
             bin_cap=20, dt_min_log2=-28, steps=20, variants=False),
        # the largest workload: every one of 16,777,216 particles active
        dict(name="zeldovich_16m_first", kind="first", ics="zeldovich", nside=256, masses="equal",
             leaf_max=16, cell_margin=2.0, bin_cap=14, dt_min_log2=-24, steps=2, variants=False),
        # the differentiation workload: 20 steps forward and back, the loss on
        # the final density on a 32^3 grid
        dict(name="gradient_33k", kind="gradient", ics="clumpy", nside=32, n_clumps=8,
             per_clump=512, masses="equal", leaf_max=8, cell_margin=2.0, bin_cap=12,
             dt_min_log2=-24, steps=20, n_grid=32, variants=False),
        # a state's density on a grid (an output or a loss) and its adjoint
        dict(name="grid_111k", kind="grid", ics="clumpy", nside=48, n_clumps=8, per_clump=1024,
             masses="equal", leaf_max=8, cell_margin=2.0, bin_cap=12, dt_min_log2=-24, steps=0,
             n_grid=64, variants=False),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["passes", "first", "run", "run", "build", "gradient", "grid"])
    c = dict(kind=kind, leaf_max=rng.choice([8, 16]), cell_margin=rng.choice([1.5, 2.0]),
             masses=rng.choice(["equal", "equal", "random"]), variants=False, steps=0)
    if kind in ("passes", "first", "build", "run"):
        c["ics"] = rng.choice(["lattice", "sedov", "clustered", "zeldovich"])
    else:
        c["ics"] = rng.choice(["clumpy", "lattice"])
    if c["ics"] == "clustered":
        spheres = rng.randint(3, 64)
        total = size(6000, 2500000)
        c.update(n_spheres=spheres, per_sphere=max(60, total // (2 * spheres)),
                 n_background=max(3000, total // 2), bin_cap=20, dt_min_log2=-28)
    else:
        top = dict(passes=100, first=200, build=200, run=128, gradient=44, grid=64)[kind]
        c.update(nside=size(14, top), bin_cap=rng.choice([0, 10, 12, 14]), dt_min_log2=-24)
        if c["ics"] == "clumpy":
            c.update(n_clumps=rng.randint(2, 12))
            c.update(per_clump=max(40, c["nside"] ** 3 // (8 * c["n_clumps"])))
        if kind == "passes" and c["bin_cap"] == 0:
            c["dt_min_log2"] = -15
    if kind in ("passes", "first"):
        c["steps"] = 1
    if kind == "run":
        c["steps"] = rng.randint(4, 32)
        c["variants"] = rng.random() < 0.25
    if kind == "gradient":
        c.update(steps=rng.randint(4, 20), n_grid=rng.randint(16, 48), masses="equal")
    if kind == "grid":
        c["n_grid"] = size(16, 128)
    return c


# --- particle sets -----------------------------------------------------------

def _count(case):
    if case["ics"] == "clustered":
        return case["n_background"] + case["n_spheres"] * case["per_sphere"]
    return case["nside"] ** 3


def _uniform(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _lattice(g, nside, jitter=0.1):
    d = 1.0 / nside
    c = (torch.arange(nside, device="cuda", dtype=torch.float64) + 0.5) * d
    pos = torch.stack(torch.meshgrid(c, c, c, indexing="ij"), dim=-1).reshape(-1, 3)
    return pos + (2.0 * _uniform(g, *pos.shape) - 1.0) * jitter * d


def _plummer(g, a, count):
    """Offsets of a Plummer sphere of scale radius a, truncated at 10 a."""
    edge = (100.0 / 101.0) ** 1.5  # mass inside 10 a
    x = _uniform(g, count) * (edge - 1e-6) + 1e-6
    r = a / torch.sqrt(x ** (-2.0 / 3.0) - 1.0)
    u = _normal(g, count, 3)
    return r[:, None] * u / u.norm(dim=1, keepdim=True)


def _plummer_density(pos, centres, radii, per_sphere):
    out = torch.zeros(pos.shape[0], device="cuda", dtype=torch.float64)
    for c, a in zip(centres, radii):
        d = pos - c
        d -= torch.round(d)
        out += 3.0 * per_sphere / (4.0 * math.pi * a ** 3) * (1.0 + (d * d).sum(1) / a ** 2) ** -2.5
    return out


def _ics(case, seed):
    """pos, vel (float64), m, u, h0 (float32) of a case's particle set."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 1000003)
    n, kind = _count(case), case["ics"]
    n_est = torch.full((n,), float(n), device="cuda", dtype=torch.float64)
    u = torch.ones(n, device="cuda", dtype=torch.float64)
    vel = torch.zeros(n, 3, device="cuda", dtype=torch.float64)
    if kind == "clustered":
        nb, ns, per = case["n_background"], case["n_spheres"], case["per_sphere"]
        centres = _uniform(g, ns, 3)
        radii = torch.exp(math.log(1e-3) + _uniform(g, ns) * math.log(30.0)).tolist()
        pos = torch.cat([_uniform(g, nb, 3)] +
                        [c + _plummer(g, a, per) for c, a in zip(centres, radii)])
        pos -= torch.floor(pos)
        n_est = nb + _plummer_density(pos, centres, radii, per)
        contrast = n_est / nb
        # thermal energies such that the time steps span 2^13
        beta = max(0.0, 2.0 * (13.0 * math.log(2.0) / math.log(float(contrast.max())) - 1.0 / 3.0))
        u[nb:] = contrast[nb:] ** beta
    elif kind == "zeldovich":
        side = case["nside"]
        d = 1.0 / side
        k1 = torch.fft.fftfreq(side, d=d, device="cuda", dtype=torch.float64) * 2.0 * math.pi
        kz = torch.fft.rfftfreq(side, d=d, device="cuda", dtype=torch.float64) * 2.0 * math.pi
        k2 = k1[:, None, None] ** 2 + k1[None, :, None] ** 2 + kz[None, None, :] ** 2
        ok = (k2 > 0) & (k2 <= (math.pi * side) ** 2)
        k2 = torch.where(ok, k2, torch.ones_like(k2))
        delta = torch.fft.rfftn(_normal(g, side, side, side)) * torch.where(
            ok, k2 ** -0.625 / k2, torch.zeros_like(k2))
        psi = torch.stack([torch.fft.irfftn(1j * k * delta, s=(side, side, side), dim=(0, 1, 2))
                           .reshape(-1) for k in (k1[:, None, None], k1[None, :, None],
                                                  kz[None, None, :])], dim=1)
        psi *= 0.3 * d / torch.sqrt((psi * psi).sum(1).mean())
        pos = _lattice(g, side, 0.0) + psi
    else:
        side = case["nside"]
        pos = _lattice(g, side)
        if kind == "sedov":
            u[:] = 1e-5
            hot = torch.argsort(((pos - 0.5) ** 2).sum(1), stable=True)[:32]
            u[hot] = n / 32.0
        elif kind == "clumpy":
            nc, per = case["n_clumps"], case["per_clump"]
            moved = torch.randperm(n, generator=g, device="cuda")[:nc * per]
            centres = _uniform(g, nc, 3)
            radii = torch.exp(math.log(1e-3) + _uniform(g, nc) * math.log(30.0)).tolist()
            for k, (c, a) in enumerate(zip(centres, radii)):
                pos[moved[k * per:(k + 1) * per]] = c + _plummer(g, a, per)
            pos -= torch.floor(pos)
            n_est = n - nc * per + _plummer_density(pos, centres, radii, per)
        else:
            vel = 0.2 * _normal(g, n, 3)  # a moving gas: the viscosity acts
    pos = pos - torch.floor(pos)
    pos = torch.where(pos >= 1.0, torch.zeros_like(pos), pos)
    m = torch.full((n,), 1.0 / n, device="cuda", dtype=torch.float64)
    if case["masses"] == "random":
        m *= 0.5 + _uniform(g, n)
    h0 = ETA * n_est ** (-1.0 / 3.0)
    return dict(pos=pos, vel=vel.float(), m=m.float(), u=u.float(), h0=h0.float(), rng=g)


def _particles(case, ic, counts=False):
    p = sim.Particles(_count(case), with_counts=counts, with_gradients=case["variants"])
    for k, name in enumerate("xyz"):
        getattr(p, name).copy_(ic["pos"][:, k])
        getattr(p, "v" + name).copy_(ic["vel"][:, k])
    p.m.copy_(ic["m"])
    p.A.copy_(ic["u"])  # holds u until the first density pass
    p.h.copy_(ic["h0"])
    return p


def _params(case):
    on = int(case["variants"])
    return sim.Params(cfl=CFL, bin_cap=case["bin_cap"], dt_min=2.0 ** case["dt_min_log2"],
                      leaf_max=case["leaf_max"], cell_margin=case["cell_margin"], balsara=on,
                      predict_inactive=on, limiter=on)


# --- the cases ---------------------------------------------------------------

def prepare(case, seed):
    ic = _ics(case, seed)
    kind = case["kind"]
    s = dict(case=dict(case), kind=kind)
    n = _count(case)
    if kind == "gradient":
        s["run"] = adjoint.Run(_params(case), ic["m"], ic["h0"], case["steps"], case["n_grid"])
        s["ic"] = [ic["pos"], ic["vel"].double(), ic["u"].double()]
        s["target"] = torch.ones(case["n_grid"] ** 3, device="cuda", dtype=torch.float64)
        return s
    s["ctx"] = sim.Context(_params(case), n)
    counts = kind == "passes"
    s["saved"] = _particles(case, ic, counts)
    if kind == "grid":
        s["saved"].ti_drift.fill_(7)  # sampled some ticks after the particles' last drift
        s["bar"] = _normal(ic["rng"], case["n_grid"] ** 3)
        s["adj"] = sim.Adjoint(n)
        return s
    s["p"] = sim.Particles(n, with_counts=counts, with_gradients=case["variants"])
    if kind in ("passes", "first"):
        s["out"] = sim.Particles(n, with_counts=counts, with_gradients=case["variants"])
    return s


GRID_TICK = 4096


def run(s):
    case, kind = s["case"], s["kind"]
    if kind == "gradient":
        pos, vel, u = (t.detach().requires_grad_(True) for t in s["ic"])
        rho = adjoint.GridDensityRun.apply(pos, vel, u, s["run"])
        loss = ((rho - s["target"]) ** 2).sum()
        loss.backward()
        return dict(rho=rho.detach(), pos=pos.grad, vel=vel.grad, u=u.grad)
    ctx, saved = s["ctx"], s["saved"]
    if kind == "grid":
        adj = s["adj"].zero_()
        rho = ctx.grid_density(saved, case["n_grid"], GRID_TICK)
        ctx.grid_density_bwd(saved, case["n_grid"], GRID_TICK, s["bar"], adj)
        return dict(rho=rho, x=adj.x, y=adj.y, z=adj.z, vx=adj.vx, vy=adj.vy, vz=adj.vz, h=adj.h)
    p = s["p"]
    ctx.state_copy(saved, p, False)
    ctx.resume(p, 0, True)
    if kind == "passes":
        ctx.build_cells(p)
        ctx.mark_active(p, 0)
        ctx.kick_drift(p, 0)
        ctx.density_active(p, 1)  # sets the entropy from u
        ctx.force_active(p)
        ctx.kick_drift(p, 1)
        ctx.timestep_bins(p)
        ctx.kick_drift(p, 2)
    elif kind == "build":
        ctx.build_cells(p)
    else:
        ctx.step_graph(p, case["steps"])
    if kind in ("passes", "first"):
        ctx.state_copy(p, s["out"], True)
        return s["out"].arrays()
    return dict(p.arrays(), perm=ctx.perm_tensor(p.n))


def work(case):
    """What a pass cannot do without: the state read once and written once, and
    the pair terms of the steps in which every particle is active (a run's first
    step, both steps of a cold set); later steps' pairs depend on the data and
    are not counted."""
    n, kind = _count(case), case["kind"]
    pairs = NGB * n
    if kind == "build":
        return dict(bytes=2 * STATE_BYTES * n, flops=0)
    if kind == "gradient":
        return dict(bytes=(28 + 28 + 56 + 56) * n + 16 * case["n_grid"] ** 3,
                    flops=pairs * (29 + 61 + 45 + 150))
    if kind == "grid":
        h = ETA * n ** (-1.0 / 3.0)
        points = n * 4.0 / 3.0 * math.pi * (GK * h * case["n_grid"]) ** 3
        return dict(bytes=2 * 52 * n + 16 * case["n_grid"] ** 3 + 56 * n, flops=points * (20 + 35))
    full = case["steps"] if kind == "first" else 1
    return dict(bytes=2 * STATE_BYTES * n, flops=pairs * (29 + 61) * full)


# --- 64-bit values -----------------------------------------------------------

def _w(q):
    return torch.where(q < 0.5, 1 - 6 * q ** 2 + 6 * q ** 3, 2 * (1 - q).clamp(min=0) ** 3)


def _dw(q):
    return torch.where(q < 0.5, -12 * q + 18 * q ** 2, -6 * (1 - q).clamp(min=0) ** 2)


def _min_image(d):
    return d - torch.round(d)


def _neighbours(pos, radius):
    """Pairs (i, j), i != j, with r_ij < max(radius_i, radius_j)."""
    ii, jj = [], []
    n = pos.shape[0]
    rows = max(1, (1 << 25) // n)
    for a in range(0, n, rows):
        r2 = torch.zeros(min(rows, n - a), n, device="cuda", dtype=torch.float64)
        for k in range(3):
            r2 += _min_image(pos[a:a + rows, k, None] - pos[None, :, k]) ** 2
        i, j = torch.nonzero(r2 < torch.maximum(radius[a:a + rows, None], radius[None, :]) ** 2,
                             as_tuple=True)
        keep = i + a != j
        ii.append(i[keep] + a)
        jj.append(j[keep])
    return torch.cat(ii), torch.cat(jj)


def _sum(i, x, n):
    return torch.zeros(n, device="cuda", dtype=torch.float64).index_add_(0, i, x)


def _exact_step(case, seed):
    ic = _ics(case, seed)
    n = _count(case)
    pos = ic["pos"]
    vel, m, u, h0 = (ic[k].double() for k in ("vel", "m", "u", "h0"))
    i, j = _neighbours(pos, 1.35 * GK * h0)
    d = _min_image(pos[i] - pos[j])
    r = d.norm(dim=1)
    lo, hi = 0.7 * h0, 1.35 * h0
    for _ in range(60):  # h^3 n(h) = eta^3, increasing in h
        h = 0.5 * (lo + hi)
        over = (1.0 + _sum(i, _w((r / (GK * h[i])).clamp(max=1.0)), n)) * KN / GK ** 3 > ETA ** 3
        hi, lo = torch.where(over, h, hi), torch.where(over, lo, h)
    h = 0.5 * (lo + hi)
    H = GK * h
    qi, qj = (r / H[i]).clamp(max=1.0), (r / H[j]).clamp(max=1.0)
    sr = m + _sum(i, m[j] * _w(qi), n)
    srt = 3 * m + _sum(i, m[j] * (3 * _w(qi) + qi * _dw(qi)), n)
    rho, f = KN * sr / H ** 3, 3 * sr / (3 * sr - srt)
    A = (GAMMA - 1) * u / rho ** (GAMMA - 1)
    P = A * rho ** GAMMA
    c = torch.sqrt(GAMMA * P / rho)
    Q = f * P / rho ** 2
    dwi, dwj = KN * _dw(qi) / H[i] ** 4, KN * _dw(qj) / H[j] ** 4
    near = r < torch.maximum(H[i], H[j])
    vr = ((vel[i] - vel[j]) * d).sum(1) / r
    wij = vr.clamp(max=0.0)
    vs = c[i] + c[j] - 3 * wij
    Pi = -ALPHA * vs * wij / (rho[i] + rho[j])
    mean = 0.5 * (dwi + dwj)
    t = m[j] * (Q[i] * dwi + Q[j] * dwj + Pi * mean) / r
    a = [_sum(i, -t * d[:, k], n) for k in range(3)]
    Adot = 0.5 * (GAMMA - 1) * rho ** (1 - GAMMA) * _sum(i, m[j] * Pi * mean * vr, n)
    vsig = (2 * c).scatter_reduce(0, i[near], vs[near], "amax")
    dt_min = 2.0 ** case["dt_min_log2"]
    bins = torch.floor(torch.log2(CFL * h / vsig / dt_min)).clamp(0, case["bin_cap"])
    half = 0.5 * 2.0 ** bins * dt_min  # the opening half-kick of the new step
    out = dict(x=pos[:, 0], y=pos[:, 1], z=pos[:, 2], ax=a[0], ay=a[1], az=a[2], A=A + Adot * half,
               Adot=Adot, h=h, rho=rho, f=f, P=P, c=c, vsig=vsig, m=m)
    for k, name in enumerate(("vx", "vy", "vz")):
        out[name] = vel[:, k] + a[k] * half
    return dict(out, bin=None, ti_begin=None, ti_end=None, ti_drift=None, active=None,
                ngb_density=None, ngb_force=None)


def _exact_grid(case, seed):
    ic = _ics(case, seed)
    n, ng = _count(case), case["n_grid"]
    bar = _normal(ic["rng"], ng ** 3).reshape(ng, ng, ng)  # [z, y, x]
    dt = (GRID_TICK - 7) * 2.0 ** case["dt_min_log2"]
    pos = ic["pos"] + ic["vel"].double() * dt
    m, h = ic["m"].double(), ic["h0"].double()
    H = GK * h
    rho = torch.zeros(ng ** 3, device="cuda", dtype=torch.float64)
    g = torch.zeros(4, n, device="cuda", dtype=torch.float64)
    order = torch.argsort(H)
    k0 = 0
    while k0 < n:  # particles of like support together: a box of points around each
        most = max(1, (1 << 24) // (2 * math.ceil(float(H[order[k0]]) * ng) + 2) ** 3)
        idx = order[k0:k0 + most]
        w = 2 * math.ceil(float(H[idx[-1]]) * ng) + 2
        idx = idx[:max(1, (1 << 24) // w ** 3)]
        k0 += idx.numel()
        w = min(w, ng)
        base = torch.floor(pos[idx] * ng).long() - w // 2
        at = base[:, :, None] + torch.arange(w, device="cuda")
        d = _min_image(pos[idx][:, :, None] - (at.double() + 0.5) / ng)
        at = at % ng
        cell = (at[:, 2, :, None, None] * ng + at[:, 1, None, :, None]) * ng + at[:, 0, None, None, :]
        r = torch.sqrt(d[:, 2, :, None, None] ** 2 + d[:, 1, None, :, None] ** 2 +
                       d[:, 0, None, None, :] ** 2)
        Hk, mk = H[idx, None, None, None], m[idx, None, None, None]
        q = (r / Hk).clamp(max=1.0)
        rho.index_add_(0, cell.reshape(-1), (mk * KN * _w(q) / Hk ** 3).reshape(-1))
        b = bar.reshape(-1)[cell]
        t = b * mk * KN * _dw(q) / Hk ** 4 / r.clamp(min=1e-300)
        g[0, idx] = (t * d[:, 0, None, None, :]).sum((1, 2, 3))
        g[1, idx] = (t * d[:, 1, None, :, None]).sum((1, 2, 3))
        g[2, idx] = (t * d[:, 2, :, None, None]).sum((1, 2, 3))
        g[3, idx] = (-b * mk * GK * KN / Hk ** 4 * (3 * _w(q) + q * _dw(q))).sum((1, 2, 3))
    return dict(rho=rho, x=g[0], y=g[1], z=g[2], vx=g[0] * dt, vy=g[1] * dt, vz=g[2] * dt, h=g[3])


def exact(case, seed):
    # larger sets would need a neighbour search of their own; later steps and
    # the clumps' h, far from its guess, a whole second implementation
    if case["kind"] in ("passes", "first") and case["ics"] == "lattice" and _count(case) <= 45000:
        return _exact_step(case, seed)
    if case["kind"] == "grid":
        return _exact_grid(case, seed)
    return None
