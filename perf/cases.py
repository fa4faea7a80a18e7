"""The work that programs have this library do, as timed cases.

A case is one call a user's program repeats: advance a particle set by whole
advection steps and read its state back, advance a batch of cases, follow an
observable step by step, or order particles that are already on the device.
``listed()`` names the cases, ``draw()`` gives others of the same ranges,
``prepare()`` makes what a program holds before the call, ``run()`` is the
call, ``work()`` what it cannot do without, and ``exact()`` what it returns in
64-bit arithmetic, from a plain restatement of the scheme in torch.
"""
import math

import numpy as np
import torch

import paper_2503_16082_gb300 as S

# fluids of the library's workloads: (drop rho, outer rho, drop eta, outer eta, sigma, c0)
FLUIDS = {
    # water-air-like drop of the static, oscillating and impacting workloads
    "heavy": (1000.0, 1.0, 0.1, 0.001, 1.0, 10.0),
    # impacting drop: Re = 1e4, We = 2.5e4
    "impact": (1000.0, 1.0, 0.1, 0.001, 0.04, 10.0),
    # equal densities, the viscous regime of the Laplace and oscillation checks
    "equal": (1.0, 1.0, 0.05, 0.05, 1.0, 20.0),
    # Couette flow around a drop, capillary number 0.1
    "shear": (1.0, 1.0, 1.0, 1.0, 1.25, 11.2),
}
WALL_LAYERS = 3


def listed():
    return [
        # the smallest call: a coarse 2D drop, as in quick studies and smoke runs
        dict(name="drop2d_f32_576", kind="drop", dim=2, n=24, precision=32, fluid="equal", box=1.0, vel=0.3, steps=1),
        # the 2D static drop followed in double precision (config of the Laplace check), 8 lanes as the notes advise
        dict(name="laplace2d_f64_6k", kind="drop", dim=2, n=80, precision=64, fluid="heavy", box=2.0, vel=0.08, steps=1,
             lanes=8, block=64),
        # the 2D oscillating drop at R = 24 dp, its observables reduced on the device after every step
        dict(name="follow2d_f64_14k", kind="drop", dim=2, n=120, precision=64, fluid="equal", box=1.0, vel=2.0, steps=1,
             lanes=4, block=64, diagnose=True),
        # the sheared drop: periodic in x, moving walls, R = 24 dp
        dict(name="shear2d_f32_37k", kind="drop", dim=2, n=192, precision=32, fluid="shear", box=8.0, vel=0.5, steps=2,
             periodic=True),
        # a 3D drop of a parameter study, library defaults
        dict(name="drop3d_f32_64k", kind="drop", dim=3, n=40, precision=32, fluid="heavy", box=2.0, vel=0.08, steps=1),
        # a ragged 3D box with the neighbour cells walked instead of listed (the option that needs no list memory)
        dict(name="cells3d_f32_30k", kind="drop", dim=3, n=31, precision=32, fluid="heavy", box=2.0, vel=0.08, steps=1,
             cells=True),
        # the 3D oscillating drop in double precision
        dict(name="drop3d_f64_43k", kind="drop", dim=3, n=35, precision=64, fluid="heavy", box=2.0, vel=0.08, steps=1),
        # the benchmark's 3D oscillating drop, a million fluid particles, its launch shape
        dict(name="drop3d_f32_1m", kind="drop", dim=3, n=100, precision=32, fluid="heavy", box=2.0, vel=0.08, steps=1,
             block=256),
        # the drop impact: the largest workload, few substeps between rebuilds
        dict(name="impact3d_f32_7m", kind="impact", dim=3, n=60, precision=32, fluid="impact", vel=1.0, steps=1),
        # a parameter study in one batch: 2D and 3D drops of mixed sizes
        dict(name="batch_f32_24", kind="batch", members=24, lo=2000, hi=60000, precision=32, steps=1),
        # cell order of particles that another program keeps on the device
        dict(name="order3d_300k", kind="order", dim=3, count=300000),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["drop", "drop", "drop", "drop", "drop", "batch", "order", "impact"])
    if kind == "order":
        return dict(kind="order", dim=rng.choice([2, 3]), count=int(_log(rng, 2000, 500000)))
    if kind == "batch":
        return dict(kind="batch", members=rng.randint(5, 30), lo=2000, hi=int(_log(rng, 6000, 60000)), precision=32,
                    steps=1)
    if kind == "impact":
        return dict(kind="impact", dim=3, n=rng.randint(12, 50), precision=32, fluid="impact", vel=1.0, steps=1)
    dim = rng.choice([2, 3])
    precision = rng.choice([32, 32, 64])
    cells = rng.random() < 0.15
    top = {(2, 32): 300, (2, 64): 160, (3, 32): 110, (3, 64): 42}[dim, precision]
    c = dict(kind="drop", dim=dim, n=int(_log(rng, 16 if dim == 3 else 20, min(top, 50) if cells else top)),
             precision=precision, steps=1)
    if dim == 2 and rng.random() < 0.3:
        c.update(fluid="shear", box=8.0, vel=0.5, periodic=True)
    elif rng.random() < 0.4:
        c.update(fluid="equal", box=1.0, vel=rng.uniform(0.3, 2.0))
    else:
        c.update(fluid="heavy", box=2.0, vel=rng.uniform(0.05, 0.15))
    if cells:
        c["cells"] = True
    elif c["n"] ** dim < 60000:
        c["lanes"] = rng.choice([1, 2, 4, 8])
    c["block"] = rng.choice([64, 128, 160, 256])
    return c


# ------------------------------------------------------------------ inputs
def _lattice(lo, hi, dx):
    axes = [a + (np.arange(int(round((b - a) / dx))) + 0.5) * dx for a, b in zip(lo, hi)]
    return np.stack([g.ravel() for g in np.meshgrid(*axes, indexing="ij")], axis=1)


def _problem(c, rng):
    """Particles and parameters of one drop: a slightly disordered lattice
    with a smooth velocity field, as a run has it once it is under way."""
    dim, n = c["dim"], c["n"]
    rho_d, rho_o, eta_d, eta_o, sigma, c0 = FLUIDS[c["fluid"]]
    impact = c["kind"] == "impact"
    hi = [4.0, 4.0, 2.0] if impact else [c["box"]] * dim
    dx = 1.0 / n if impact else c["box"] / n
    lo = [0.0] * dim
    p = _lattice(lo, hi, dx)
    center = np.array([2.0, 2.0, 0.6]) if impact else np.array(hi) / 2
    # R = 0.5 in the impact, a quarter of the box in the drops, an eighth in the shear flow; a mode-2 surface
    R = 0.5 if impact else hi[0] * (0.125 if c.get("periodic") else 0.25)
    d = p - center
    r2 = (d * d).sum(axis=1)
    amp = 0.0 if impact else 0.05 * c.get("amp", 1.0)
    cos2 = np.where(r2 > 0, d[:, -1] ** 2 / np.where(r2 > 0, r2, 1.0), 0.0)
    drop = r2 < (R * (1.0 + amp * (1.5 * cos2 - 0.5))) ** 2
    p += rng.uniform(-0.02, 0.02, p.shape) * dx
    # every axis's velocity varies along the next one, so the field has no divergence
    v = np.empty_like(p)
    for a in range(dim):
        x = p[:, (a + 1) % dim] * (2 * math.pi / hi[(a + 1) % dim])
        v[:, a] = (0.05 if impact else 0.2 if c.get("periodic") else 1.0) * c["vel"] * np.sin(x + rng.uniform(0, 2 * math.pi))
    periodic = 1 if c.get("periodic") else 0
    if impact:
        v[drop, 2] -= c["vel"]
    if periodic:
        v[:, 0] += c["vel"] * (2 * p[:, 1] / hi[1] - 1)
        p[:, 0] = np.mod(p[:, 0], hi[0])
    big_lo = [-WALL_LAYERS * dx if not (periodic >> a) & 1 else 0.0 for a in range(dim)]
    w = _lattice(big_lo, [hi[a] - big_lo[a] for a in range(dim)], dx)
    w = w[~np.all((w > 0.0) & (w < np.array(hi)), axis=1)]
    walls = [(w, [0.0] * 3)]
    if periodic:
        walls = [(w[w[:, 1] < 0], [-c["vel"], 0.0, 0.0]), (w[w[:, 1] > 0], [c["vel"], 0.0, 0.0])]
    return dict(dim=dim, dx=dx, c0=c0, sigma=sigma, cfl=0.4 if dim == 3 else 0.6, periodic=periodic, hi=hi,
                rho0=(rho_d, rho_o), eta=(eta_d, eta_o), fluids=[(p[drop], v[drop]), (p[~drop], v[~drop])], walls=walls)


def _members(c, rng):
    """The members of a batch: drops of both dimensions, log-uniform sizes
    that belong to the case; the particles' disorder and motion are `rng`'s."""
    out = []
    study = np.random.default_rng([c["members"], c["lo"], c["hi"]])
    for i in range(c["members"]):
        dim = 2 + i % 2
        target = math.exp(study.uniform(math.log(c["lo"]), math.log(c["hi"])))
        m = dict(kind="drop", dim=dim, n=max(8, int(round(target ** (1.0 / dim)))), fluid="heavy",
                 box=study.uniform(0.8, 2.0), vel=0.08, amp=study.uniform(0.0, 4.0))
        q = _problem(m, rng)
        q.update(sigma=math.exp(study.uniform(math.log(0.3), math.log(3.0))), cfl=0.4)
        out.append(q)
    return out


def _handle(q, c):
    par = S.default_params(dim=q["dim"], precision=c["precision"], dx=q["dx"], c0=q["c0"], gamma=q["sigma"],
                           cfl_ac=q["cfl"], periodic=q["periodic"], lanes=c.get("lanes", 1), block=c.get("block", 128),
                           nbr_mode=S.NBR_CELLS if c.get("cells") else S.NBR_LIST)
    for a in range(q["dim"]):
        par.period_lo[a], par.period_hi[a] = 0.0, q["hi"][a]
    h = S.create_case(par)
    for k, (p, v) in enumerate(q["fluids"]):
        S.add_phase_particles(h, S.FLUID, p, rho0=q["rho0"][k], eta=q["eta"][k], vel=v)
    for p, wv in q["walls"]:
        S.add_phase_particles(h, S.WALL, p, wall_vel=wv)
    return h


class State:
    """Handles and read-back buffers of one program; released with it."""

    def __init__(self, c):
        self.case, self.handles, self.batch = c, [], None

    def __del__(self):
        for h in self.handles:
            if self.batch is not None:
                S.batch_remove(self.batch, h)
            S.destroy(h)
        if self.batch is not None:
            S.batch_destroy(self.batch)


FIELDS = (("pos", S.FIELD_POS), ("vel", S.FIELD_VEL), ("rho", S.FIELD_RHO))


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    s = State(case)
    if case["kind"] == "order":
        # points in a box of cells that hold about 18 (3D) or 7 (2D) of them
        dim, n = case["dim"], case["count"]
        m = max(3, int((n / (18.0 if dim == 3 else 7.0)) ** (1.0 / dim)))
        s.ncell = [m] * dim
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        s.pos = torch.rand((n, 3), generator=g, dtype=torch.float64, device="cuda") * (m * 0.999)
        s.keys = torch.empty(n, dtype=torch.int64, device="cuda")
        s.order = torch.empty(n, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        return s
    probs = _members(case, rng) if case["kind"] == "batch" else [_problem(case, rng)]
    s.handles = [_handle(q, case) for q in probs]
    s.dims = [q["dim"] for q in probs]
    if case["kind"] == "batch":
        s.batch = S.batch_create(case["precision"])
        for h in s.handles:
            S.batch_add(s.batch, h)
        S.batch_step(s.batch, 0)        # places the members on the device
    else:
        S.step(s.handles[0], 0)         # places the case on the device
    # pinned read-back buffers, one per field, all members one after the other
    s.views, s.flat, s.single = [], [], []
    for name, f in FIELDS:
        sizes = [S.num_particles(h)[0] * (d if f in S.VECTOR_FIELDS else 1) for h, d in zip(s.handles, s.dims)]
        buf = torch.empty(sum(sizes), dtype=torch.float64, pin_memory=True)
        s.views.append(np.split(buf.numpy(), np.cumsum(sizes)[:-1]))
        s.flat.append(buf)
        # the values of a 32-bit run, kept as the program stores them
        s.single.append(torch.empty(sum(sizes), dtype=torch.float32) if case["precision"] == 32 else None)
    return s


def run(state):
    c = state.case
    if c["kind"] == "order":
        S.cell_order_noalloc(c["dim"], c["count"], state.pos.data_ptr(), [0.0] * c["dim"], 1.0, state.ncell,
                             state.keys.data_ptr(), state.order.data_ptr(), torch.cuda.current_stream().cuda_stream)
        return {"keys": state.keys, "order": state.order}
    if state.batch is not None:
        S.batch_step(state.batch, c["steps"])
    else:
        S.step(state.handles[0], c["steps"])
    out = {}
    for (name, f), views, flat, single in zip(FIELDS, state.views, state.flat, state.single):
        for h, d, v in zip(state.handles, state.dims, views):
            S.read_fields(h, f, d, out=v)
        out[name] = flat if single is None else single.copy_(flat)
    if c.get("diagnose"):
        q = S.diagnose(state.handles[0], center=(c["box"] / 2, c["box"] / 2), r_in=c["box"] / 8, r_out=c["box"] * 0.4)
        out["shape"] = np.array(q["second"][:2] + q["first"][:2] + [q["kinetic"]])
        out["inside"] = q["n_in"]
    return out


# -------------------------------------------------------------------- work
def _count(c):
    """(particles, fluid particles, neighbours, substeps) of one drop."""
    dim, n = c["dim"], c["n"]
    dx = 1.0 / n if c["kind"] == "impact" else c["box"] / n
    fluid = (4 * n) * (4 * n) * (2 * n) if c["kind"] == "impact" else n ** dim
    shell = ((4 * n + 6) ** 2 * (2 * n + 6) if c["kind"] == "impact"
             else (n + 6) * n if c.get("periodic") else (n + 6) ** dim)
    h = 1.3 * dx
    rho, eta, sigma, c0 = FLUIDS[c["fluid"]][:2], FLUIDS[c["fluid"]][2:4], FLUIDS[c["fluid"]][4], FLUIDS[c["fluid"]][5]
    v = max(c["vel"], 1e-3)
    ad = 0.1 * min([h / v] + [r * h * h / e for r, e in zip(rho, eta)])
    ac = (0.4 if dim == 3 else 0.6) * min([h / (c0 + v)] + [math.sqrt(r * h ** 3 / (2 * math.pi * sigma)) for r in rho])
    return shell, fluid, (80 if dim == 3 else 20), max(1, math.ceil(ad / ac))


def work(case):
    if case["kind"] == "order":
        return {"bytes": case["count"] * (24 + 8 + 8), "flops": 0}
    if case["kind"] == "batch":
        # the expected member: the mean of a log-uniform size, half of them 2D
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        one = [work(dict(kind="drop", dim=d, n=max(8, round(mean ** (1.0 / d))), precision=case["precision"], fluid="heavy",
                         box=1.4, vel=0.08, steps=case["steps"])) for d in (2, 3)]
        return {k: case["members"] * (one[0][k] + one[1][k]) / 2 for k in ("bytes", "flops")}
    total, fluid, nbr, subs = _count(case)
    size = case["precision"] // 8
    # a substep reads and writes position, velocity and density of each fluid particle once and reads its frozen
    # position and viscous acceleration; each pair takes about 59 operations of pressure and 35 of continuity, and
    # 85 of viscosity, correction and shift once per step; the state is read back in 64 bits
    d = case["dim"]
    by = case["steps"] * subs * fluid * size * (2 * (2 * d + 1) + 2 * d) + total * (2 * d + 1) * 8
    fl = case["steps"] * fluid * nbr * (subs * (59 + 35) + 85)
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------- exact
def _pairs(q, x, fluid, h, chunk=1 << 20):
    """Neighbours j of fluid particles i with 0 < r < 2h: chunks of
    (i0, i1, i - i0, j, e, W', r), i ascending."""
    dim, dev = q["dim"], x.device
    cs0 = 2 * h * (1 + 1e-6)
    lo = x.min(0).values - 0.5 * cs0
    m = torch.clamp(((x.max(0).values - lo) / cs0).long() + 1, min=1)
    width = torch.full((dim,), cs0, dtype=x.dtype, device=dev)
    L = q["hi"][0]
    if q["periodic"]:
        lo[0], m[0] = 0.0, int(L / cs0)
        width[0] = L / int(m[0])
    cell = torch.minimum(((x - lo) / width).long(), m - 1)
    strides = torch.ones(dim, dtype=torch.long, device=dev)
    for a in range(1, dim):
        strides[a] = strides[a - 1] * m[a - 1]
    ncell = int(torch.prod(m))
    key = (cell * strides).sum(1)
    skey, order = torch.sort(key)
    start = torch.searchsorted(skey, torch.arange(ncell + 1, device=dev))
    alpha = 7 / (4 * math.pi * h * h) if dim == 2 else 21 / (16 * math.pi * h ** 3)
    out = []
    for i0 in range(0, fluid, chunk):
        i1 = min(fluid, i0 + chunk)
        ii, jj = [], []
        for o in np.ndindex(*([3] * dim)):
            cc = cell[i0:i1] + (torch.tensor(o, device=dev) - 1)
            if q["periodic"]:
                cc[:, 0] %= m[0]
            ok = ((cc >= 0) & (cc < m)).all(1)
            k = torch.where(ok, (cc * strides).sum(1), torch.zeros_like(ok, dtype=torch.long))
            cnt = torch.where(ok, start[k + 1] - start[k], torch.zeros_like(k))
            i = torch.repeat_interleave(torch.arange(i0, i1, device=dev), cnt)
            first = torch.repeat_interleave(start[k] - (torch.cumsum(cnt, 0) - cnt), cnt)
            j = order[first + torch.arange(len(i), device=dev)]
            rv = x[i] - x[j]
            if q["periodic"]:
                rv[:, 0] -= L * torch.round(rv[:, 0] / L)
            r2 = (rv * rv).sum(1)
            keep = (r2 < 4 * h * h) & (i != j)
            ii.append(i[keep])
            jj.append(j[keep])
        i, j = torch.cat(ii), torch.cat(jj)
        i, at = torch.sort(i, stable=True)
        j = j[at]
        rv = x[i] - x[j]
        if q["periodic"]:
            rv[:, 0] -= L * torch.round(rv[:, 0] / L)
        r = rv.square().sum(1).sqrt()
        u = r / h
        out.append((i0, i1, i - i0, j, rv / r[:, None], -5 * alpha / h * u * (1 - 0.5 * u) ** 3, r))
    return out


def _sum(v, i, n):
    return torch.zeros((n,) + v.shape[1:], dtype=v.dtype, device=v.device).index_add_(0, i, v)


def _advance(q, steps, dev):
    """The scheme of the paper in 64 bits: state after `steps` advection
    steps, particles in the order they were added."""
    dim, dx, c0, gam = q["dim"], q["dx"], q["c0"], q["sigma"]
    h, vol = 1.3 * dx, dx ** dim
    T = dict(dtype=torch.float64, device=dev)
    x = torch.tensor(np.concatenate([p for p, _ in q["fluids"]] + [p for p, _ in q["walls"]]), **T)
    v = torch.tensor(np.concatenate([w for _, w in q["fluids"]] + [np.tile(np.array(wv)[:dim], (len(p), 1))
                                                                   for p, wv in q["walls"]]), **T)
    n0, nf, n = len(q["fluids"][0][0]), sum(len(p) for p, _ in q["fluids"]), len(x)
    kind = torch.full((n,), 2, dtype=torch.long, device=dev)
    kind[:n0], kind[n0:nf] = 0, 1
    rho0 = torch.tensor([q["rho0"][0], q["rho0"][1], q["rho0"][0]], **T)
    eta = torch.tensor([q["eta"][0], q["eta"][1], 0.0], **T)
    ref, mass = rho0[kind], rho0[kind] * vol
    dr = torch.zeros(n, **T)          # density deviation
    xi = 1.3 * math.log10(max(q["rho0"]) / min(q["rho0"])) + 0.6
    ph = torch.tensor([q["rho0"][k] / sum(q["rho0"]) for k in (0, 1)], **T)
    lo = torch.zeros(dim, **T)

    def top(k):
        w = v[:n0] if k == 0 else v[n0:nf]
        return math.sqrt(float(w.square().sum(1).max())) if len(w) else 0.0

    for _ in range(steps):
        if q["periodic"]:
            x[:, 0] = lo[0] + torch.remainder(x[:, 0] - lo[0], q["hi"][0])
        vm = [top(k) for k in (0, 1)]
        dt_ad = min(0.1 * min([q["rho0"][k] * h * h / q["eta"][k]] + ([h / vm[k]] if vm[k] > 0 else [])) for k in (0, 1))
        pairs = _pairs(q, x, nf, h)
        V = torch.where(kind == 2, torch.full_like(ref, vol), mass / (ref + dr))
        B = torch.zeros((n, dim, dim), **T)
        eye = torch.eye(dim, **T)
        for i0, i1, i, j, e, dw, r in pairs:
            M = torch.empty((i1 - i0, dim, dim), **T)
            for a in range(dim):
                for b in range(a, dim):
                    M[:, a, b] = M[:, b, a] = _sum(dw * V[j] * r * e[:, a] * e[:, b], i, i1 - i0)
            bad = torch.linalg.det(M).abs() < 1e-3
            M[bad] = -eye
            B[i0:i1] = -torch.linalg.inv(M)
        av, shift = torch.zeros((nf, dim), **T), torch.zeros((nf, dim), **T)
        for i0, i1, i, j, e, dw, r in pairs:
            g = i + i0
            wall = kind[j] == 2
            ei, ej = eta[kind[g]], eta[kind[j]]
            eb = torch.where(wall, ei, 2 * ei * ej / (ei + ej))
            f = (eb * dw * V[j] / r)[:, None] * (v[g] - v[j])
            av[i0:i1] = 2 / (ref + dr)[i0:i1, None] * _sum(f, i, i1 - i0)
            ew = e * (dw * V[j])[:, None]
            part = torch.where(wall[:, None], torch.einsum("pab,pb->pa", B[g], ew), torch.einsum("pab,pb->pa", B[j], ew))
            shift[i0:i1] = _sum(part, i, i1 - i0) + torch.einsum("pab,pb->pa", B[i0:i1], _sum(ew, i, i1 - i0))
        x[:nf] -= 0.2 * h * h * shift
        t_in = 0.0
        while True:
            vm = [top(k) for k in (0, 1)]
            dt_ac = min(q["cfl"] * min(h / (c0 + vm[k]), math.sqrt(q["rho0"][k] * h ** 3 / (2 * math.pi * gam))) for k in (0, 1))
            last = dt_ac >= dt_ad - t_in
            dt = dt_ad - t_in if last else dt_ac
            rho = ref + dr
            p = c0 * c0 * dr
            V = torch.where(kind == 2, torch.full_like(ref, vol), mass / rho)
            gc = torch.zeros((n, dim), **T)
            for i0, i1, i, j, e, dw, r in pairs:
                sel = (kind[i + i0] + kind[j]) == 1
                g, jj = (i + i0)[sel], j[sel]
                w = 2 * ph[kind[g]] * dw[sel] * V[jj]
                gc[i0:i1] = _sum(w[:, None] * e[sel], i[sel], i1 - i0)
            gn = gc.square().sum(1).sqrt()
            on = gn * h > 1e-4
            nh = torch.where(on[:, None], gc / torch.where(on, gn, torch.ones_like(gn))[:, None], torch.zeros_like(gc))
            acc = torch.empty((nf, dim), **T)
            for i0, i1, i, j, e, dw, r in pairs:
                g = i + i0
                wall = kind[j] == 2
                ri, rj, pi, pj = rho[g], rho[j], p[g], p[j]
                du = ((v[j] - v[g]) * e).sum(1)
                du = torch.where(wall, 2 * du, du)
                beta = torch.clamp(3 * du / c0, 0.0, 1.0)
                ps = torch.where(wall, pi + 0.5 * beta * ri * c0 * du,
                                 (ri * pj + rj * pi + beta * c0 * ri * rj * du) / (ri + rj))
                f = -2 * _sum((ps * V[j] * dw)[:, None] * e, i, i1 - i0)
                # surface stress and penalty of the pairs that touch the interface
                sel = ~wall & ((gn[g] > 0) | (gn[j] > 0))
                g, jj, ee, w, rr = g[sel], j[sel], e[sel], dw[sel] * V[j[sel]], r[sel]
                same = (kind[g] == kind[jj])[:, None]
                ni, nj = nh[g], nh[jj]
                pe = lambda a, m: gam * (torch.where(on[a], gn[a], torch.zeros_like(gn[a])))[:, None] * (  # noqa: E731
                    ee - m * (m * ee).sum(1, keepdim=True))
                Pi, Pj = pe(g, ni), pe(jj, nj)
                bar = 0.5 * torch.where(same, gc[g] + gc[jj], gc[g] - gc[jj])
                bn = bar.square().sum(1, keepdim=True).sqrt()
                fac = rr[:, None] * (bar * ee).sum(1, keepdim=True) / torch.where(bn > 0, bn, torch.ones_like(bn))
                c = torch.where(same, torch.zeros_like(ee), ee) - fac * bar
                nc = 0.5 * (ni * (ni * c).sum(1, keepdim=True) + nj * (nj * c).sum(1, keepdim=True))
                pen = (xi * gam / rr)[:, None]
                a, b = ph[kind[g]][:, None], ph[kind[jj]][:, None]
                s = torch.where(same, Pi + Pj + pen * (c - nc), 2 * b * Pi + 2 * a * Pj - 4 * a * b * pen * nc)
                f += _sum(s * w[:, None], i[sel], i1 - i0)
                acc[i0:i1] = f / rho[i0:i1, None]
            v[:nf] += dt * (acc + av)
            rate = torch.empty(nf, **T)
            for i0, i1, i, j, e, dw, r in pairs:
                g = i + i0
                dve = ((v[g] - v[j]) * e).sum(1)
                rel = torch.where(kind[j] == 2, dve, (rho[j] * c0 * dve + p[g] - p[j]) / (c0 * (rho[g] + rho[j])))
                rate[i0:i1] = 2 * rho[i0:i1] * _sum(rel * V[j] * dw, i, i1 - i0)
            dr[:nf] += dt * rate
            x[:nf] += dt * v[:nf]
            t_in += dt
            if last:
                break
    return x, v, torch.where(kind == 2, rho0[0], ref + dr), n0


def exact(case, seed):
    if case["kind"] == "order":
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    rng = np.random.default_rng(seed)
    probs = _members(case, rng) if case["kind"] == "batch" else [_problem(case, rng)]
    got = [_advance(q, case["steps"], dev) for q in probs]
    out = {name: torch.cat([g[k].reshape(-1) for g in got]) for k, (name, _) in enumerate(FIELDS)}
    if case.get("diagnose"):
        x, v, _, n0 = got[0]
        m = torch.tensor(probs[0]["rho0"], dtype=torch.float64, device=dev) * probs[0]["dx"] ** case["dim"]
        nf = sum(len(p) for p, _ in probs[0]["fluids"])
        kin = 0.5 * (m[0] * v[:n0].square().sum() + m[1] * v[n0:nf].square().sum())
        out["shape"] = torch.cat([x[:n0].square().sum(0), x[:n0].sum(0), kin.reshape(1)])
        out["inside"] = None
    return out
