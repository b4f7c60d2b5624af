"""What a user of the framework has it do, as timed cases.

A case is one call (or the short sequence of calls) that a simulation makes
again and again: a force evaluation, a kick-drift-kick step, the gradient of a
density loss through a step, an ensemble's graph launch, the placement of
positions into the particle layout.  The layouts are the repository's own: one
PM level of twice the particle lattice; the two-level run (meshes of half and
of twice the lattice); the isolated two-level run (half and four times).
Particles are synthetic, made on the GPU from a seed: a Zel'dovich field of a
BBKS spectrum, and for the evolved states a share of the particles in haloes
(a power law of masses, NFW profiles of 200 times the mean density, centred on
the field's own particles; with 0.55 of the particles about the 200 pairs in
range per particle and the cell counts that the 256^3 run ends with).

``exact`` is the same mathematics in 64 bits with plain torch: the optimised
Green's function by its image sum, FFT solves, the 4-point difference, the
pair forces over the 27 neighbouring cells.
"""
import math

import numpy as np
import torch

from paper_2512_12629_gb300 import cube2

OM, OL, HUBBLE, SIGMA8 = 0.3, 0.7, 0.7, 0.8
FIX = 65536
LATTICES = (12, 16, 24, 32, 48, 64, 96, 128, 192, 256)


def _case(name, kind, n, layout="two", z=49.0, haloes=0.0, missing=0, order=2, fp16=False, pm3=False, boxes=0,
          persistent=False):
    """kind: force, step, gradient, ensemble or place.  n: lattice (= cells of the particle layout) per side,
    the particle count is n^3 - missing.  haloes: the share of particles in haloes.  order: 2 CIC, 3 TSC."""
    return dict(name=name, kind=kind, n=n, layout=layout, z=z, haloes=haloes, missing=missing, order=order, fp16=fp16,
                pm3=pm3, boxes=boxes, persistent=persistent)


def listed():
    return [
        # the smallest box of the repository: one force, where launches and latency count
        _case("force-32", "force", 32, "one"),
        # the same recipe as the large runs at a size for parameter studies: one step
        _case("step-64-mid", "step", 64, z=1.0, haloes=0.2),
        # the main run (256^3, 128^3 + 512^3 meshes): a step at its start, one particle per cell
        _case("step-256-early", "step", 256),
        # the main run near its end: dense cells, most of the time in pairs
        _case("step-256-late", "step", 256, z=0.02, haloes=0.55),
        # radix-3 meshes and a particle count that is no cube, half way through a run
        _case("force-192-ragged", "force", 192, z=2.0, haloes=0.15, missing=123457),
        # the paper's own assignment (TSC) on an evolved state
        _case("force-128-tsc", "force", 128, z=0.5, haloes=0.4, order=3),
        # isolated boundary conditions, fine mesh of four times the lattice
        _case("force-64-isolated", "force", 64, "iso", z=0.0, haloes=0.5, missing=1001),
        # the differentiation workload: loss and gradient through one step
        _case("gradient-128", "gradient", 128, "one", z=1.0, haloes=0.1),
        # the large workload's layout at an eighth of its volume, FP16 velocities
        _case("step-512-fp16", "step", 512, z=1.0, fp16=True),
        # many independent small boxes in one graph launch
        _case("ensemble-16", "ensemble", 0, "one", boxes=16, z=3.0),
        # arbitrary positions into the particle layout: the entry of a differentiable run
        _case("place-128", "place", 128, z=1.0, haloes=0.2, missing=54321),
        # the adaptive third level on an evolved state
        _case("force-128-pm3", "force", 128, z=0.0, haloes=0.5, pm3=True),
    ]


def draw(rng):
    kind = rng.choice(["force", "force", "step", "step", "step", "gradient", "ensemble", "place"])
    if kind == "ensemble":
        return _draw_done(_case("", kind, 0, "one", z=rng.uniform(1.0, 49.0), boxes=rng.randint(3, 24),
                                persistent=rng.random() < 0.5))
    z = rng.choice([49.0, rng.uniform(0.0, 6.0), rng.uniform(0.0, 1.0)])
    haloes = 0.0 if z > 6 else rng.uniform(0.0, 0.6) / (1.0 + z)
    layout = rng.choice(["one", "two", "two", "iso"]) if kind in ("force", "step") else rng.choice(["one", "two"])
    top = 96 if layout == "iso" else 128 if kind == "gradient" else 256
    n = rng.choice([v for v in LATTICES if v <= top and (v >= 16 or layout == "one")])
    missing = rng.choice([0, rng.randint(1, max(1, n ** 3 // 20))])
    order = 3 if kind in ("force", "step") and rng.random() < 0.2 else 2
    pm3 = kind == "force" and layout == "two" and order == 2 and n >= 48 and n != 12 and rng.random() < 0.3
    fp16 = kind == "step" and rng.random() < 0.25
    return _draw_done(_case("", kind, n, layout, z, haloes, missing, order, fp16, pm3))


def _draw_done(c):
    del c["name"]
    return c


# ------------------------------------------------------------ configuration
def _count(case):
    return case["n"] ** 3 - case["missing"]


def _levels(n, layout):
    """((mesh, beta), ...) coarsest first, box side [Mpc/h]."""
    if layout == "one":
        return ((2 * n, 2.0),), 2.0 * n
    if layout == "two":
        return ((n // 2, 3.5), (2 * n, 2.0)), 1.0 * n
    return ((n // 2, 3.5), (4 * n, 3.5)), 2.0 * n


def _config(n, layout, count, order=2, fp16=False, pm3=False):
    levels, box = _levels(n, layout)
    c = cube2.Config()
    c.box, c.n_ios, c.n_levels = box, n, len(levels)
    for i, (mesh, beta) in enumerate(levels):
        c.n_mesh[i], c.beta[i] = mesh, beta
    c.b_pp = 0.1 * box / n
    c.omega_m, c.omega_l = OM, OL
    c.n_particles = count
    c.alias_max = 2
    c.assign_order = order
    c.iso_length = 0.5 * box if layout == "iso" else 0.0
    c.vel_fp16 = int(fp16)
    if pm3:   # the repository's calibration: subtiles of 8^3 cells, twice the resolution, 2 cells softening
        c.pm3_tile, c.pm3_refine, c.pm3_beta, c.pm3_rho_min, c.pm3_max_tiles = 8, 2, 2.0, 512, 512
    return c


def _context(cfg):
    ctx = cube2.init_mesh(cfg)
    for level in range(cfg.n_levels):
        cube2.set_green(ctx, level)
    if cfg.pm3_tile > 0:
        cube2.set_green(ctx, cube2.LEVEL_PM3)
    return ctx


def _schedule(case):
    """One step of the 50-step schedule (z = 49 to 0) from the case's redshift."""
    a0 = 1.0 / (1.0 + case["z"])
    return [a0, a0 + 0.0196]


# ---------------------------------------------------------------- particles
def _hubble(a):
    return np.sqrt(OM * np.asarray(a, dtype=np.float64) ** -3 + OL)


def _integral(a0, a1, power):
    x, w = np.polynomial.legendre.leggauss(48)
    a = 0.5 * (a0 + a1) + 0.5 * (a1 - a0) * x
    return float(0.5 * (a1 - a0) * np.sum(w / (a ** power * _hubble(a))))


def _growth(a):
    def d(t):
        s = np.linspace(1e-4, t, 20001)
        f = (s * _hubble(s)) ** -3
        return float(_hubble(t) * np.sum(0.5 * (f[1:] + f[:-1]) * np.diff(s)))
    return d(a) / d(1.0)


def _transfer(k):
    q = k / (OM * HUBBLE)
    poly = 1.0 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3 + (6.71 * q) ** 4
    return (torch.log1p(2.34 * q) / (2.34 * q) if torch.is_tensor(q) else np.log1p(2.34 * q) / (2.34 * q)) * poly ** -0.25


def _amplitude():
    k = np.exp(np.linspace(math.log(1e-5), math.log(1e2), 20001))
    x = 8.0 * k
    w = 3.0 * (np.sin(x) - x * np.cos(x)) / x ** 3
    f = k ** 4 * _transfer(k) ** 2 * w * w / (2.0 * math.pi ** 2)
    return SIGMA8 ** 2 / float(np.sum(0.5 * (f[1:] + f[:-1]) * np.diff(np.log(k))))


def _raw(n, box, z, haloes, missing, seed):
    """Unsorted particles: positions (3, N) in cells (FP64), momenta and forces (3, N) FP32."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    a = 1.0 / (1.0 + z)
    d = _growth(a)
    cell = box / n
    dk = torch.fft.rfftn(torch.randn((n, n, n), generator=gen, device=dev))
    kf = 2.0 * math.pi / box
    k1 = torch.fft.fftfreq(n, d=1.0 / n, device=dev) * kf
    k = (k1[None, None, :n // 2 + 1].abs(), k1[None, :, None], k1[:, None, None])
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    k2[0, 0, 0] = 1.0
    kk = torch.sqrt(k2)
    dk *= torch.sqrt(_amplitude() * kk * _transfer(kk) ** 2 * (n / box) ** 3) / k2
    dk[0, 0, 0] = 0.0
    del k2, kk
    q = torch.arange(n, device=dev, dtype=torch.float64) + 0.5
    grid = (q[None, None, :], q[None, :, None], q[:, None, None])
    pos = torch.empty((3, n, n, n), dtype=torch.float64, device=dev)
    acc = torch.empty((3, n, n, n), dtype=torch.float32, device=dev)
    for i in range(3):
        acc[i] = torch.fft.irfftn(1j * k[i] * dk, s=(n, n, n)) * d      # D psi, the linear force, Mpc/h
        pos[i] = grid[i] + acc[i].double() / cell
    del dk
    pos, acc = pos.view(3, -1), acc.view(3, -1)
    if missing or haloes > 0.0:
        pick = torch.randperm(n ** 3, generator=gen, device=dev)[: n ** 3 - missing]
        pos, acc = pos[:, pick], acc[:, pick]
        del pick
    vel = acc * float(a * a * _hubble(a) * (OM * a ** -3 / _hubble(a) ** 2) ** 0.55)
    if haloes > 0.0:
        _add_haloes(pos, vel, acc, int(haloes * pos.shape[1]), a, cell, gen)
    return pos, vel, acc


def _add_haloes(pos, vel, acc, members, a, cell, gen):
    """The first `members` particles moved into NFW haloes (mass in particles: one per cell at the mean density)."""
    dev = pos.device
    lo, hi, s = 16.0, max(64.0, min(8.0e3, members / 8.0)), -1.3
    u = torch.rand(members // 16 + 1, generator=gen, device=dev, dtype=torch.float64)
    mass = torch.floor((lo ** s + u * (hi ** s - lo ** s)) ** (1.0 / s)).long()
    owner = torch.repeat_interleave(torch.arange(mass.numel(), device=dev), mass)[:members]
    mass = mass.double()
    centre = pos[:, torch.randint(members, pos.shape[1], (mass.numel(),), generator=gen, device=dev)]
    rvir = (3.0 * mass / (4.0 * math.pi * 200.0)) ** (1.0 / 3.0)
    conc = 4.0
    t = torch.linspace(0.0, 1.0, 8193, device=dev, dtype=torch.float64)
    enclosed = torch.log1p(conc * t) - conc * t / (1.0 + conc * t)
    enclosed = enclosed / enclosed[-1]
    frac = torch.rand(owner.numel(), generator=gen, device=dev, dtype=torch.float64)
    r = t[torch.searchsorted(enclosed, frac).clamp(max=8192)] * rvir[owner]
    way = torch.randn((3, owner.numel()), generator=gen, device=dev, dtype=torch.float64)
    way /= way.norm(dim=0, keepdim=True)
    m = owner.numel()
    pos[:, :m] = centre[:, owner] + r * way
    pull = mass[owner] * frac / (4.0 * math.pi * torch.clamp(r, min=0.1) ** 2) * cell
    acc[:, :m] = (-pull * way).float()
    # virial motions: about a tenth of a cell per step in a halo of a thousand particles
    drift = _integral(a, a + 0.0196, 3)
    speed = 0.1 * cell / drift * (mass[owner] / 1000.0) ** (1.0 / 3.0)
    vel[:, :m] += (speed * torch.randn((3, m), generator=gen, device=dev, dtype=torch.float64)).float()


def _cells(fixed, n):
    c = fixed >> 16
    return (c[2] * n + c[1]) * n + c[0]


def _sorted(pos, vel, acc, n):
    """The particle layout: sorted by cell, 16-bit offsets in the cell, counts and starts."""
    fixed = torch.remainder(torch.round(pos * FIX).long(), n * FIX)
    cell = _cells(fixed, n).to(torch.int32)
    cell, order = torch.sort(cell, stable=True)
    off = torch.stack([(fixed[i] & (FIX - 1)).to(torch.int32).to(torch.int16)[order] for i in range(3)])
    count = torch.bincount(cell, minlength=n ** 3).to(torch.int32)
    start = (torch.cumsum(count, 0, dtype=torch.int64) - count).to(torch.int32)
    return cube2.IOSState(off, count, start, torch.stack([v[order] for v in vel]), torch.stack([f[order] for f in acc]))


def _state(case, seed):
    n = case["n"]
    box = _levels(n, case["layout"])[1]
    return _sorted(*_raw(n, box, case["z"], case["haloes"], case["missing"], seed), n)


def _target(case, seed):
    """A target density: plain CIC of another realisation on the finest mesh."""
    n = case["n"]
    (levels, box) = _levels(n, case["layout"])
    mesh = levels[-1][0]
    pos = _raw(n, box, case["z"], 0.0, 0, seed + 7919)[0]
    rho = _deposit(pos * (mesh / n), mesh, 2) - 1.0
    return rho.float()


BOX_SIZES = (32, 48, 32, 64, 32, 48, 24, 96)


def _box_sizes(case):
    return [BOX_SIZES[b % len(BOX_SIZES)] for b in range(case["boxes"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        return _prepare_ensemble(case, seed)
    n = case["n"]
    ctx = _context(_config(n, case["layout"], _count(case), case["order"], case["fp16"], case["pm3"]))
    s = dict(case=case, ctx=ctx)
    if kind == "place":
        box = _levels(n, case["layout"])[1]
        pos, vel, _ = _raw(n, box, case["z"], case["haloes"], case["missing"], seed)
        s.update(pos=pos * (box / n), mom=vel.contiguous())
        return s
    p = _state(case, seed)
    if case["fp16"]:
        ctx.vel_encode(p, p.vel)
        p.vel = p.vel[:, :1].clone()   # unused with FP16 storage
    s.update(p=p, a=_schedule(case))
    if kind == "gradient":
        cube2.adjoint_init(ctx)
        s["target"] = _target(case, seed)
    return s


def _prepare_ensemble(case, seed):
    """All boxes' particles in one tensor per field: what a study that replays its graph from many initial states
    keeps, so that one copy per field brings in the next states."""
    sizes = _box_sizes(case)
    made = [_sorted(*_raw(n, 2.0 * n, case["z"], 0.0, 0, seed * 1000 + b), n) for b, n in enumerate(sizes)]
    first, work, states = [], [], [[] for _ in sizes]
    for field in ("off", "count", "start", "vel", "acc"):
        parts = [getattr(m, field) for m in made]
        flat = torch.cat([x.reshape(-1) for x in parts])
        mine = flat.clone()
        at = 0
        for b, x in enumerate(parts):
            states[b].append(mine[at:at + x.numel()].view(x.shape))
            at += x.numel()
        first.append(flat)
        work.append(mine)
    states = [cube2.IOSState(*fields) for fields in states]
    ctxs = [_context(_config(n, "one", n ** 3)) for n in sizes]
    a = np.array([_schedule(case)] * len(sizes))
    torch.cuda.synchronize()
    opts = cube2.ensemble_opts(n_streams=16, persistent_pp=case["persistent"])
    ens = cube2.Ensemble(ctxs, states, a, opts=opts)
    return dict(case=case, ens=ens, first=first, work=work)


def run(state):
    kind = state["case"]["kind"]
    if kind == "ensemble":
        for dst, src in zip(state["work"], state["first"]):
            dst.copy_(src)
        state["ens"].launch()
        return dict(zip(("off", "count", "start", "vel", "acc"), state["work"]))
    ctx = state["ctx"]
    if kind == "place":
        p, perm = cube2.ios_from_positions(ctx, state["pos"], state["mom"])
        return dict(off=p.off, count=p.count, start=p.start, vel=p.vel, perm=perm)
    p, a = state["p"], state["a"]
    if kind == "force":
        cube2.force(ctx, p)
        return dict(acc=p.acc)
    if kind == "gradient":
        loss, dx, dv = cube2.loss_gradient(ctx, p, state["target"], a)
        return dict(loss=loss, dx=dx, dv=dv)
    q = p.clone()   # the step works in place; a run keeps the state before it as its checkpoint
    cube2.kdk_step(ctx, q, a[0], a[1])
    out = dict(off=q.off, count=q.count, start=q.start, acc=q.acc)
    if state["case"]["fp16"]:
        out.update(vel=q.vel16.view(torch.float16), scale=q.vscale)
    else:
        out["vel"] = q.vel
    return out


# --------------------------------------------------------------------- work
def work(case):
    """Bytes: the inputs read once and the outputs written once.  Flops: the transforms of every level (a real
    transform each way), and 30 for each ordered pair in range: 4 pi / 3 per particle where the density is even,
    and about 330 more per particle in a halo."""
    kind = case["kind"]
    if kind == "ensemble":
        per = [work(_case("", "step", n, "one", z=case["z"])) for n in _box_sizes(case)]
        return {k: float(sum(w[k] for w in per)) for k in ("bytes", "flops")}
    n, N = case["n"], _count(case)
    cells = n ** 3
    if kind == "place":
        return {"bytes": float(N * (24 + 12 + 6 + 12 + 4) + 8 * cells), "flops": float(10 * N)}
    levels, box = _levels(n, case["layout"])
    fft = sum(2 * 2.5 * m ** 3 * math.log2(m ** 3) for m, _ in levels)
    reach = levels[-1][1] * box / levels[-1][0] * n / box
    pair = 30.0 * N * (4.0 * math.pi / 3.0 * reach ** 3 + 330.0 * case["haloes"])
    green = sum(4.0 * (m // 2 + 1) ** 3 / 6.0 for m, _ in levels)
    if kind == "force":
        return {"bytes": N * 18.0 + 8.0 * cells + green, "flops": fft + pair + 200.0 * N}
    if kind == "gradient":   # the step forward, and two products: each two solves per level and the pairs' Jacobian
        mesh = 4.0 * levels[-1][0] ** 3
        return {"bytes": N * (18.0 + 12.0 + 24.0) + 8.0 * cells + green + mesh, "flops": 5 * fft + 4 * pair + 1000.0 * N}
    v = 6.0 if case["fp16"] else 12.0
    scale = 8.0 * cells if case["fp16"] else 0.0
    return {"bytes": N * 2 * (6.0 + v + 12.0) + 16.0 * cells + scale + green, "flops": fft + pair + 250.0 * N}


# ---------------------------------------------------------- 64-bit reference
def _profile(k, b):
    """Eq. (Sk): the transform of the softened profile."""
    x = 0.5 * k * b
    small = x < 0.5
    xs = torch.where(small, x, torch.zeros_like(x)) ** 2
    series = torch.zeros_like(x)
    for j in range(13, 1, -1):
        series = series * xs + (-1) ** j * (2 * j - 2) / math.factorial(2 * j)
    xl = torch.where(small, torch.ones_like(x), x)
    return 12.0 * torch.where(small, series, (2.0 - 2.0 * torch.cos(xl) - xl * torch.sin(xl)) / xl ** 4)


def _green(n, soft, trunc, order, iso):
    """Eq. (Gk) for all |m| <= n/2 by the image sum |n_d| <= 2, expanded to the half spectrum [kz][ky][kx]."""
    dev = torch.device("cuda")
    m = torch.arange(n // 2 + 1, device=dev, dtype=torch.float64)
    k = 2.0 * math.pi / n * m
    fd = 4.0 / 3.0 * torch.sin(k) - 1.0 / 6.0 * torch.sin(2.0 * k)
    fd[n // 2] = 0.0
    axis = [lambda t: t[None, None, :], lambda t: t[None, :, None], lambda t: t[:, None, None]]
    images = [k + 2.0 * math.pi * i for i in range(-2, 3)]
    window = [torch.sinc(q / (2.0 * math.pi)) ** (2 * order) for q in images]
    num = torch.zeros((n // 2 + 1,) * 3, device=dev, dtype=torch.float64)
    den = torch.zeros_like(num)
    for iz in range(5):
        for iy in range(5):
            for ix in range(5):
                q = [axis[d](images[i]) for d, i in enumerate((ix, iy, iz))]
                w2 = axis[0](window[ix]) * axis[1](window[iy]) * axis[2](window[iz])
                k2 = q[0] ** 2 + q[1] ** 2 + q[2] ** 2
                k2 = torch.where(k2 > 0, k2, torch.ones_like(k2))
                kk = torch.sqrt(k2)
                s2 = _profile(kk, soft) ** 2
                if trunc is not None:
                    s2 = s2 - _profile(kk, trunc) ** 2
                if iso:
                    x = kk * iso
                    s2 = s2 * torch.where(x < 1e-2, x * x / 6.0 - x ** 4 / 120.0, 1.0 - torch.sin(x) / x)
                dot = axis[0](fd) * q[0] + axis[1](fd) * q[1] + axis[2](fd) * q[2]
                num -= w2 * dot * s2 / k2
                den += w2
    d2 = axis[0](fd) ** 2 + axis[1](fd) ** 2 + axis[2](fd) ** 2
    g = torch.where(d2 > 0, num / (torch.where(d2 > 0, d2, torch.ones_like(d2)) * den ** 2), torch.zeros_like(num))
    i = torch.arange(n, device=dev)
    i = torch.minimum(i, n - i)
    return g[i][:, i]


def _corners(u, n, order):
    """(flat mesh index, weight) of each corner of the clouds at u (3, K) mesh cells."""
    if order == 2:
        i0 = torch.floor(u.detach() - 0.5)
        f = u - 0.5 - i0
        w = (1.0 - f, f)
    else:
        i0 = torch.floor(u.detach())
        f = u - i0 - 0.5
        w = (0.5 * (0.5 - f) ** 2, 0.75 - f ** 2, 0.5 * (0.5 + f) ** 2)
        i0 = i0 - 1
    i = [torch.remainder(i0.long() + j, n) for j in range(order)]
    for z in range(order):
        for y in range(order):
            for x in range(order):
                yield (i[z][2] * n + i[y][1]) * n + i[x][0], w[z][2] * w[y][1] * w[x][0]


def _deposit(u, n, order):
    """Mean-one density of positions u (3, N) in mesh cells (FP64)."""
    rho = torch.zeros(n ** 3, dtype=torch.float64, device=u.device)
    for idx, w in _corners(u, n, order):
        rho = rho.index_add(0, idx, w)
    return (rho * (n ** 3 / u.shape[1])).view(n, n, n)


def _difference(phi):
    """The 4-point difference along x, y, z (one at a time)."""
    for axis in (2, 1, 0):
        yield 2.0 / 3.0 * (phi.roll(-1, axis) - phi.roll(1, axis)) - 1.0 / 12.0 * (phi.roll(-2, axis) - phi.roll(2, axis))


def _gather(field, u, n, order):
    f = field.reshape(-1)
    return sum(w * f[idx] for idx, w in _corners(u, n, order))


def _fixed(p, n):
    """Fixed-point coordinates (3, N) in 2^-16 cells of a state."""
    c = torch.repeat_interleave(torch.arange(n ** 3, device=p.off.device), p.count.long())
    c = torch.stack([c % n, (c // n) % n, c // (n * n)])
    return c * FIX + (p.off.long() & (FIX - 1))


def _mesh_cells(X, n, mesh):
    """Positions in mesh cells, floored to 2^-16 of one."""
    return (torch.div(X * mesh, n, rounding_mode="floor")).double() / FIX


def _tables(case):
    """Per level: (mesh, H, Green's table)."""
    levels, box = _levels(case["n"], case["layout"])
    out, prev = [], None
    for l, (mesh, beta) in enumerate(levels):
        H = box / mesh
        iso = 0.5 * box / H if case["layout"] == "iso" and l == 0 else 0.0
        out.append((mesh, H, _green(mesh, beta, None if prev is None else prev / H, case["order"], iso)))
        prev = beta * H
    return out, prev, box


def _mesh_force(case, X, tables):
    F = torch.zeros(X.shape, dtype=torch.float64, device=X.device)
    for mesh, H, g in tables:
        u = _mesh_cells(X, case["n"], mesh)
        phi = torch.fft.irfftn(torch.fft.rfftn(_deposit(u, mesh, case["order"]) - 1.0) * g, s=(mesh,) * 3)
        for d, e in enumerate(_difference(phi)):
            F[d] -= H * _gather(e, u, mesh, case["order"])
    return F


def _reference_force(r, b):
    """Eq. (refforce)."""
    u = r / b
    inner = 64 / 5 * u - 256 / 5 * u ** 3 + 32 * u ** 4 + 1536 / 35 * u ** 5 - 192 / 5 * u ** 6
    shell = (3 / 35 / u ** 2 - 32 / 5 + 256 / 5 * u - 96 * u ** 2 + 256 / 5 * u ** 3 + 32 * u ** 4 - 1536 / 35 * u ** 5
             + 64 / 5 * u ** 6)
    return torch.where(u < 0.5, inner, torch.where(u < 1.0, shell, 1.0 / u ** 2)) / b ** 2


def _pairs(X, count, n, reach, term, chunk=1 << 25):
    """Sum of term(d, i, j) over the pairs with 0 < |d| < reach (cells; a number or one per particle), d = x_j - x_i
    (3, K), for every particle i: (3, N)."""
    dev = X.device
    N = X.shape[1]
    x = X.double() / FIX
    c = X >> 16
    count = count.long()
    start = torch.cumsum(count, 0) - count
    r2max = torch.as_tensor(reach, dtype=torch.float64, device=dev).expand(N) ** 2
    F = torch.zeros((3, N), dtype=torch.float64, device=dev)
    zero = torch.zeros(1, dtype=torch.float64, device=dev)
    for k in range(27):
        s = (k % 3 - 1, (k // 3) % 3 - 1, k // 9 - 1)
        q = [torch.remainder(c[d] + s[d], n) for d in range(3)]
        cell = (q[2] * n + q[1]) * n + q[0]
        num, beg = count[cell], start[cell]
        ends = torch.cumsum(num, 0)
        lo, done = 0, 0
        while lo < N:
            hi = int(torch.searchsorted(ends, done + chunk, right=True))
            hi = max(hi, lo + 1)
            part = num[lo:hi]
            i = torch.repeat_interleave(torch.arange(lo, hi, device=dev), part)
            j = beg[i] + torch.arange(i.numel(), device=dev) - (ends - num)[i] + done
            d = torch.stack([x[a, j] - x[a, i] for a in range(3)])
            for a in range(3):   # the periodic image that lies in the neighbouring cell
                d[a] -= n * torch.round(d[a] / n)
            r2 = (d * d).sum(0)
            keep = torch.nonzero((r2 > 0) & (r2 < r2max[i])).squeeze(1)
            f = term(d[:, keep], i[keep], j[keep])
            last = torch.cumsum(torch.bincount(i[keep] - lo, minlength=hi - lo), 0)
            for a in range(3):
                run_sum = torch.cat([zero, torch.cumsum(f[a], 0)])[last]
                F[a, lo:hi] += run_sum - torch.cat([zero, run_sum[:-1]])
            done = int(ends[hi - 1])
            lo = hi
    return F


def _pair_force(case, X, count, reach_cells, box):
    n = case["n"]
    coef = n ** 3 / X.shape[1] / (4.0 * math.pi) * (box / n)
    ranges = torch.as_tensor(reach_cells, dtype=torch.float64, device=X.device).expand(X.shape[1])

    def term(d, i, j):
        r = torch.sqrt((d * d).sum(0))
        return coef * (_reference_force(r, 0.1) - _reference_force(r, ranges[i])) / r * d
    return _pairs(X, count, n, ranges, term)


def _third_level(case, X, count, F, b_fine, box):
    """Adds the local meshes' force to F; returns the pair range (cells) of every particle."""
    n, T = case["n"], 8
    cell = box / n
    H3 = box / (2 * n) / 2
    b3, B = 2.0 * H3, int(math.ceil(b_fine / H3 - 1e-12)) + 4
    need = T * 4 + 2 * B
    m = min(2 ** a * 3 ** b for a in range(9) for b in range(6) if 2 ** a * 3 ** b >= need)
    g = _green(m, 2.0, b_fine / H3, 2, 0.0)
    ns = n // T
    dense = count.view(ns, T, ns, T, ns, T).amax((1, 3, 5)) >= 512
    reach = torch.full((X.shape[1],), b_fine / cell, dtype=torch.float64, device=X.device)
    for sz, sy, sx in torch.nonzero(dense)[:512].tolist():
        origin = torch.tensor([[sx], [sy], [sz]], device=X.device) * T * FIX - B * (FIX // 4)
        rel = torch.remainder(X - origin, n * FIX)
        src = (rel < m * FIX // 4).all(0)
        own = ((rel >= B * FIX // 4) & (rel < (B + 4 * T) * FIX // 4)).all(0)
        u = rel[:, src].double() * 4 / FIX
        rho = torch.zeros(m ** 3, dtype=torch.float64, device=X.device)
        for idx, w in _corners(u, m, 2):
            rho.index_add_(0, idx, w)
        rho = rho.view(m, m, m) * (box ** 3 / X.shape[1] / H3 ** 3)
        phi = torch.fft.irfftn(torch.fft.rfftn(rho) * g, s=(m, m, m))
        u = rel[:, own].double() * 4 / FIX
        for d, e in enumerate(_difference(phi)):
            F[d, own] -= H3 * _gather(e, u, m, 2)
        reach[own] = b3 / cell
    return reach


def _force(case, X, count):
    tables, b_fine, box = _tables(case)
    F = _mesh_force(case, X, tables)
    reach = b_fine / (box / case["n"])
    if case["pm3"]:
        reach = _third_level(case, X, count, F, b_fine, box)
    return F + _pair_force(case, X, count, reach, box)


def _single(x):
    return np.float32(x).astype(np.float64)


def _moved(case, p):
    """Kick and drift of a state with the layout's 32-bit momenta and fixed-point positions, sorted again:
    (momenta FP64 of FP32 values, coordinates, counts, order)."""
    n = case["n"]
    box = _levels(n, case["layout"])[1]
    a0, a1 = _schedule(case)
    kick = _single(1.5 * OM * _integral(a0, 0.5 * (a0 + a1), 2))
    drift = _single(_integral(a0, a1, 3) * FIX / (box / n))
    v = (p.vel.double() + kick * p.acc.double()).float()
    X = _fixed(p, n)
    X = torch.remainder(X + torch.round((v.double() * drift).float()).long(), n * FIX)
    cell, order = torch.sort(_cells(X, n), stable=True)
    count = torch.bincount(cell, minlength=n ** 3)
    return v[:, order].double(), X[:, order], count, order


def _step(case, p):
    v, X, count, _ = _moved(case, p)
    F = _force(case, X, count)
    a0, a1 = _schedule(case)
    return v + 1.5 * OM * _integral(0.5 * (a0 + a1), a1, 2) * F, F


def _product(case, X, count, v, tables, b_fine, box):
    """d<v, F(x)>/dx: the mesh part by differentiating the deposit and the gather, the pairs by their Jacobian."""
    n = case["n"]
    out = torch.zeros_like(v)
    for mesh, H, g in tables:
        with torch.enable_grad():
            x = torch.zeros_like(v, requires_grad=True)
            u = _mesh_cells(X, n, mesh) + x / H
            phi = torch.fft.irfftn(torch.fft.rfftn(_deposit(u, mesh, 2) - 1.0) * g, s=(mesh,) * 3)
            s = sum((-H * _gather(e, u, mesh, 2) * v[d]).sum() for d, e in enumerate(_difference(phi)))
            out += torch.autograd.grad(s, x)[0]
    cell = box / n
    coef = n ** 3 / X.shape[1] / (4.0 * math.pi)
    reach = torch.tensor(b_fine / cell, dtype=torch.float64, device=X.device)

    def term(d, i, j):
        dv = v[:, j] - v[:, i]
        with torch.enable_grad():
            t = d.clone().requires_grad_(True)
            r = torch.sqrt((t * t).sum(0))
            f = coef * (_reference_force(r, 0.1) - _reference_force(r, reach)) / r * t
            return torch.autograd.grad((f * dv).sum(), t)[0]
    return out + _pairs(X, count, n, reach, term, chunk=1 << 23)


def _gradient(case, p, target):
    n = case["n"]
    a0, a1 = _schedule(case)
    v, X, count, order = _moved(case, p)
    tables, b_fine, box = _tables(case)
    mesh, H = tables[-1][:2]
    with torch.enable_grad():
        x = torch.zeros_like(v, requires_grad=True)
        delta = _deposit(_mesh_cells(X, n, mesh) + x / H, mesh, 2) - 1.0
        loss = ((delta - target.double()) ** 2).mean()
        after = torch.autograd.grad(loss, x)[0]
    dx = torch.empty_like(after)
    dx[:, order] = after
    dv = _integral(a0, a1, 3) * dx
    kick = 1.5 * OM * _integral(a0, 0.5 * (a0 + a1), 2)
    dx = dx + kick * _product(case, _fixed(p, n), p.count, dv, tables, b_fine, box)
    return loss.detach(), dx, dv


def exact(case, seed):
    with torch.no_grad():
        kind = case["kind"]
        if kind == "ensemble":
            vel, acc = [], []
            for b, n in enumerate(_box_sizes(case)):
                one = _case("", "step", n, "one", z=case["z"])
                p = _sorted(*_raw(n, 2.0 * n, case["z"], 0.0, 0, seed * 1000 + b), n)
                v, f = _step(one, p)
                vel.append(v.reshape(-1))
                acc.append(f.reshape(-1))
            return dict(off=None, count=None, start=None, vel=torch.cat(vel), acc=torch.cat(acc))
        n = case["n"]
        if n > 256 or (n == 256 and case["layout"] == "iso"):
            return None   # 64-bit meshes of 1024^3 take longer
        if kind == "place":
            box = _levels(n, case["layout"])[1]
            pos, vel, _ = _raw(n, box, case["z"], case["haloes"], case["missing"], seed)
            X = torch.remainder(torch.round(pos * (box / n) / (box / n) * FIX).long(), n * FIX)
            order = torch.sort(_cells(X, n), stable=True)[1]
            return dict(off=None, count=None, start=None, vel=vel[:, order].double(), perm=None)
        p = _state(case, seed)
        if kind == "force":
            return dict(acc=_force(case, _fixed(p, n), p.count))
        if kind == "gradient":
            loss, dx, dv = _gradient(case, p, _target(case, seed))
            return dict(loss=loss, dx=dx, dv=dv)
        if case["fp16"]:   # 16-bit codes: the momenta are those of the 32-bit step no longer
            return None
        v, F = _step(case, p)
        return dict(off=None, count=None, start=None, acc=F, vel=v)
