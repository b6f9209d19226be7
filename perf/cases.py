"""What a program that uses this library has it do, as cases that can be timed.

A case is a dict of plain values; `prepare` makes what the program has in hand before the
call (a loaded handle, a batch, device arrays), `run` is one pass through the public
binding, `work` the bytes and operations a pass cannot do without and `exact` the same
outputs from plain torch in 64 bits.

The inputs are dense beds near rest, the state a run spends its time in: a disordered
packing with small overlaps, slow random velocities and spins, ids in random order (a mixed
bed), in a box, in the lower half of a rotating drum, or above the slit of a hopper. A lid
rests on the bed, so that it keeps its 4 to 7 contacts per sphere however many passes are
timed. They are made on the GPU from the seed alone. Velocities, spins, forces and torques of an FP32 run are 32-bit values inside the
library, so `run` hands them on as float32 (no rounding); positions are double there too.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1301_1714_gb300 import dem, scenes

R0 = 1e-3        # mean radius [m]
KN = 1e4         # [N/m]
E_REST = 0.7     # restitution that sets alpha

# ------------------------------------------------------------------------- cases
_DEFAULT = dict(kind="step", shape="box", n=2048, steps=20, precision="fp32", model="practical", stiffness="linear",
                terms=0, resort=0, skin=0.15, spread=0.1, mu=0.5, block=0, slots=0, scenes=1)


def _case(**kw):
    bad = set(kw) - set(_DEFAULT) - {"name"}
    assert not bad, bad
    return {**_DEFAULT, **kw}


def listed():
    return [
        # the smallest call in earnest: the FP64 box of the parity runs, sorting every step
        _case(name="box2k_fp64_walk", n=2048, steps=20, precision="fp64", resort=1, skin=0.0, spread=0.05, mu=0.3),
        # one small request of a serving program: a few thousand spheres, Hertz law, many steps between looks
        _case(name="box9k_fp32_hertz", n=9217, steps=100, stiffness="hertz", skin=0.2, mu=0.3),
        # the polydisperse box in FP32 lists, the ordinary run, ...
        _case(name="bed262k_fp32", n=262144, steps=40, skin=0.12, spread=0.2, mu=0.3),
        # ... and the same in FP64, the run that others are checked against
        _case(name="bed262k_fp64", n=262144, steps=10, precision="fp64", skin=0.12, spread=0.2, mu=0.3),
        # the draining box of the paper's benchmark, run in chunks until at rest (never reached here)
        _case(name="hopper131k_until", kind="until", shape="hopper", n=131072, steps=50, spread=0.05, skin=0.1),
        # the largest: the drum at its full size, list mode as the autotuner sets it
        _case(name="drum4m_fp32", shape="drum", n=4194304, steps=20, block=128, slots=24),
        # the paper's own policy, sort every step, on a million spheres
        _case(name="drum1m_fp32_walk", shape="drum", n=1000003, steps=10, resort=1, skin=0.0, slots=24),
        # the simple model, the other column of the paper's tables
        _case(name="drum500k_simple", shape="drum", n=500009, steps=20, model="simple", block=128),
        # every optional force term on, Hertz stiffness, an odd size
        _case(name="bed100k_terms", n=100003, steps=20, stiffness="hertz", terms=15, mu=0.4),
        # forces on positions that come from elsewhere: load, sort and one force evaluation, no step
        _case(name="forces65k_fp64", kind="forces", n=65537, steps=1, precision="fp64", resort=1, skin=0.0, mu=0.3),
        # many uneven scenes advanced together
        _case(name="batch64_fp32", kind="batch", n=6000, scenes=64, steps=40, skin=0.2, block=128),
        # cell map and sort for a caller that may not allocate
        _case(name="sort200k_static", kind="sort", n=200003, steps=1, precision="fp64", resort=1, skin=0.0),
    ]


def _size(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return n | 1 if rng.random() < 0.7 else n


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["until", "forces", "batch", "sort"])
    if kind == "sort":
        return _case(kind="sort", n=_size(rng, 1000, 262144), steps=1, precision="fp64", resort=1, skin=0.0)
    prec = rng.choice(["fp32", "fp32", "fp64"])
    walk = rng.random() < 0.3
    mu = round(rng.uniform(0.1, 0.6), 3)
    spread = rng.choice([0.05, 0.1, 0.2])
    skin = 0.0 if walk else round(rng.uniform(0.08, 0.25), 3)
    stiff = rng.choice(["linear", "linear", "hertz"])
    block = rng.choice([0, 0, 128, 64, 96, 256])
    if kind == "batch":
        return _case(kind="batch", n=_size(rng, 1024, 8192), scenes=rng.randint(3, 64), steps=rng.randint(20, 50),
                     precision="fp32", skin=0.0 if walk else 0.2, resort=1 if walk else 0, mu=mu, block=block,
                     stiffness=stiff)
    if kind == "until":
        return _case(kind="until", shape="hopper", n=_size(rng, 4096, 200000), steps=rng.randint(20, 60), spread=0.05,
                     skin=skin, resort=1 if walk else 0, mu=mu, precision=prec, block=block)
    model = rng.choice(["practical", "practical", "practical", "simple"])
    terms = rng.choice([0, 0, 0, 1, 2, 4, 8, 15]) if model == "practical" else 0
    if kind == "forces":
        return _case(kind="forces", n=_size(rng, 1024, 300000), steps=1, precision=prec, resort=1 if walk else 0,
                     skin=skin, spread=spread, mu=mu, model=model, stiffness=stiff, terms=terms, block=block)
    n = _size(rng, 1024, 300000 if prec == "fp64" else 2000000)
    steps = rng.randint(4, 12) if n > (100000 if prec == "fp64" else 300000) else rng.randint(10, 50)
    return _case(kind="step", shape=rng.choice(["box", "drum"]), n=n, steps=steps, precision=prec, model=model,
                 stiffness=stiff, terms=terms, resort=1 if walk else 0, skin=skin, spread=spread, mu=mu, block=block)


# ------------------------------------------------------------------------ inputs
def _bed(layers_for, spread, gen, dims):
    """Spheres of radius R0 (1 +- spread) in a disordered dense packing over a floor of
    dims = (x, y) [m]: face-centred sites about a diameter apart, displaced at
    random, then pushed apart where they overlap. layers_for(sites per layer pair) is the
    number of layer pairs. Returns x, r and the plane (0 = lowest) of every site; the
    outermost sites lie 0.95 R0 inside dims and above z = 0."""
    dev = "cuda"
    a = 2.0 * R0 * (1.007 + 0.12 * spread)
    edge = 0.95 * R0
    nx, ny = (max(2, int(round((d - 2.0 * edge) / a + 0.5))) for d in dims)
    ax, ay = ((d - 2.0 * edge) / (k - 0.5) for d, k in zip(dims, (nx, ny)))
    c = a * math.sqrt(2.0) * (a * a / (ax * ay))              # the same volume per site at any width
    nz = layers_for(2 * nx * ny, c)
    shape = (2, nz, ny, nx)
    b = torch.arange(2, device=dev).reshape(2, 1, 1, 1).double() * 0.5
    gx = torch.arange(nx, device=dev).double().reshape(1, 1, 1, nx)
    gy = torch.arange(ny, device=dev).double().reshape(1, 1, ny, 1)
    gz = torch.arange(nz, device=dev).double().reshape(1, nz, 1, 1)
    r = (R0 * (1.0 + spread * (2.0 * torch.rand(shape, generator=gen, device=dev) - 1.0))).float()
    u = (0.08 * R0 * torch.randn((3,) + shape, generator=gen, device=dev)).clamp_(-0.2 * R0, 0.2 * R0)
    # the twelve nearest sites as shifts of the site array: half of them, the others mirrored
    near = [(0, 0, 0, 1), (0, 0, 1, 0)] + [(1, dz, dy, dx) for dz in (0, 1) for dy in (0, 1) for dx in (0, 1)]
    for _ in range(40):
        push = torch.zeros_like(u)
        for s, dz, dy, dx in near:
            # within a sub-lattice, or sub-lattice 1 against the eight sites of 0 around it
            for i, j in (((0, 0), (1, 1)) if s == 0 else ((1, 0),)):
                at = [(dx - 0.5 * s) * ax, (dy - 0.5 * s) * ay, (dz - 0.5 * s) * c]
                d = torch.roll(u[:, j], (-dz, -dy, -dx), (-3, -2, -1)) - u[:, i]
                d += torch.tensor(at, device=dev).float().reshape(3, 1, 1, 1)
                dist = d.square().sum(0).sqrt()
                gap = (r[i] + torch.roll(r[j], (-dz, -dy, -dx), (-3, -2, -1)) - dist).clamp_(min=0.0)
                f = d * (0.15 * gap / dist)
                push[:, i] -= f
                push[:, j] += torch.roll(f, (dz, dy, dx), (-3, -2, -1))
        u += push
    x = torch.stack([((gx + b) * ax + edge).expand(shape), ((gy + b) * ay + edge).expand(shape),
                     ((gz + b) * c + edge).expand(shape)], 0) + u.double()
    plane = (2 * gz + 2 * b).long().expand(shape).reshape(-1)
    return x.reshape(3, -1).t().contiguous(), r.reshape(-1), plane, 0.5 * c


def _pick(cand, n, gen):
    """n of the candidates in random order (the sites left out are vacancies)."""
    return cand[torch.randperm(len(cand), generator=gen, device="cuda")[:n]]


def _motion(n, gen, vs=0.03, ws=5.0):
    v = vs * torch.randn((n, 3), generator=gen, device="cuda", dtype=torch.float64)
    w = ws * torch.randn((n, 3), generator=gen, device="cuda", dtype=torch.float64)
    return v, w


def _params(case, r, lo, hi, walls, mu, e=E_REST):
    rmax = float(r.max())
    rmin = float(r.min())
    m = scenes.sphere_mass(rmin)
    alpha = scenes.alpha_from_e(e)
    eta = alpha * math.sqrt(KN * 0.5 * scenes.sphere_mass(R0))
    cn, ct = scenes.hertz_coeffs(KN, 2.0 / 7.0, R0)
    skin = case["skin"] * rmax
    return scenes.Params(
        model=case["model"], stiffness=case["stiffness"], precision=case["precision"],
        dt=scenes.linear_contact_time(KN, e, 0.5 * m) / 50.0, kn=KN, kt=KN * 2.0 / 7.0, cn=cn, ct=ct, alpha=alpha,
        mu=mu, ksp=KN, kda=eta, ksh=eta, skin=skin, cell_size=scenes.auto_cell_size(rmax, skin), domain_lo=lo,
        domain_hi=hi, resort_interval=case["resort"], terms=case["terms"], mu_roll=0.02 if case["terms"] & 2 else 0.0,
        alpha_t=0.2 if case["terms"] & 4 else 0.0, k_coh=2e3 if case["terms"] & 8 else 0.0,
        walls=[scenes._norm_wall(w) for w in walls])


def _scene(case, seed, n=None, mu=None, e=E_REST):
    """Device arrays x, v, w, r and the parameters of one scene of the case."""
    n = case["n"] if n is None else n
    mu = case["mu"] if mu is None else mu
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    spread = case["spread"]
    if case["shape"] == "drum":
        # the lower half of a drum of radius 300 : length 208, sized for n spheres
        s = (n / 4194304.0) ** (1.0 / 3.0)
        Rd = 1.045 * 300.0 * R0 * s + 2.0 * R0
        L = max(208.0 * R0 * s, 8.8 * R0)
        x, r, plane, dz = _bed(lambda per, c: int(1.25 * Rd / c) + 2, spread, gen, (L, 2.0 * Rd))
        x[:, 1] -= Rd
        x[:, 2] -= Rd
        rr = r.double()
        inside = (x[:, 1].square() + x[:, 2].square()).sqrt() + 0.95 * rr < Rd
        full = torch.cumsum(torch.bincount(plane[inside]), 0)
        top = int(torch.searchsorted(full, n))
        keep = _pick(torch.nonzero(inside & (plane <= top)).reshape(-1), n, gen)
        assert len(keep) == n, (len(keep), n)
        x, r = x[keep], r[keep]
        lid = -Rd + 1.9 * R0 + top * dz
        walls = scenes.drum_walls(Rd, L, 2.0) + [dict(kind="plane", p=(0.0, 0.0, lid), n=(0.0, 0.0, -1.0))]
        lo, hi = (0.0, -Rd, -Rd), (L, Rd, Rd)
        v, w = _motion(n, gen)
        v[:, 1] -= 2.0 * x[:, 2]                                 # the bed turns with the drum
        v[:, 2] += 2.0 * x[:, 1]
    else:
        side = max(8.4 * R0, (n * 5.6 * R0 ** 3) ** (1.0 / 3.0) * (1.0 if n < 100000 else 1.2))
        x, r, plane, dz = _bed(lambda per, c: -(-n // per), spread, gen, (side, side))
        keep = _pick(torch.arange(len(r), device="cuda"), n, gen)
        top = int(plane.max())
        x, r = x[keep], r[keep]
        z0 = 0.0
        if case["shape"] == "hopper":
            z0 = math.ceil(0.9 * top * dz / R0) * R0
            x[:, 2] += z0
        lid = z0 + 1.9 * R0 + top * dz
        lo, hi = (0.0, 0.0, 0.0), (side, side, lid)
        walls = scenes.box_walls(lo, hi)
        if case["shape"] == "hopper":
            walls += scenes.slit_plates(z0, 0.5 * side, 6.0 * R0)
        v, w = _motion(n, gen)
    return x.contiguous(), v, w, r.contiguous(), _params(case, r, lo, hi, walls, mu, e)


def _batch_scenes(case, seed):
    """Sizes from n/4 to 2n, friction and restitution of each scene (the same for every seed)."""
    rng = np.random.RandomState(case["n"] * 64 + case["scenes"])
    out = []
    for k in range(case["scenes"]):
        n = int(case["n"] * math.exp(rng.uniform(math.log(0.25), math.log(2.0))))
        out.append(_scene(case, int(seed) * 131 + k, n=n, mu=rng.uniform(0.1, 0.6), e=rng.uniform(0.5, 0.95)))
    return out


def _grid(p):
    return p.domain_lo, p.cell_size, scenes.grid_dims(p.domain_lo, p.domain_hi, p.cell_size)


def prepare(case, seed):
    st = {"case": case}
    stream = torch.cuda.Stream()
    st["stream"] = stream
    n = case["n"]
    if case["kind"] == "batch":
        sc = _batch_scenes(case, seed)
        b = _Batch(case, sc, stream)
        st["batch"] = b
        n = b.total
    else:
        x, v, w, r, p = _scene(case, seed)
        torch.cuda.synchronize()
        if case["kind"] == "sort":
            o, h, d = _grid(p)
            st.update(x=x, origin=o, cell=h, dims=d, cell_of=torch.empty(n, dtype=torch.int32, device="cuda"),
                      order=torch.empty(n, dtype=torch.int32, device="cuda"),
                      start=torch.empty(d[0] * d[1] * d[2] + 1, dtype=torch.int32, device="cuda"))
            return st
        st["sim"] = dem.Simulation(p, x, v, w, r, cuda_stream=stream.cuda_stream, block_size=case["block"],
                                   max_contacts=case["slots"])
        if case["kind"] == "forces":
            st["in"] = (x, v, w, r)
    st["out"] = [torch.empty((n, 3), dtype=torch.float64, device="cuda") for _ in range(3)]
    torch.cuda.synchronize()
    return st


class _Batch:
    """A batch and its slots; destroyed with its last reference."""

    def __init__(self, case, sc, stream):
        self.b = dem.dem_batch_create(precision=case["precision"], model=case["model"], stiffness=case["stiffness"],
                                      block_size=case["block"], cuda_stream=stream.cuda_stream)
        self.slots, self.total = [], 0
        for x, v, w, r, p in sc:
            k = dem.dem_batch_add(self.b, p, x.cpu().numpy(), v.cpu().numpy(), w.cpu().numpy(), r.cpu().numpy(),
                                  1 << 40)
            self.slots.append((k, self.total, len(r)))
            self.total += len(r)

    def __del__(self):
        dem.dem_batch_destroy(self.b)


def _typed(case, outs):
    """Velocities, spins, forces and torques of an FP32 run as the 32-bit values they are."""
    return [o.float() for o in outs] if case["precision"] == "fp32" else list(outs)


def run(st):
    case = st["case"]
    if case["kind"] == "sort":
        dem.dem_sort_cells_static(st["x"], st["origin"], st["cell"], st["dims"], st["cell_of"], st["order"],
                                  st["start"], st["stream"].cuda_stream)
        st["stream"].synchronize()      # the caller's own stream: the sort only enqueues
        return {"cell": st["cell_of"], "order": st["order"], "start": st["start"]}
    x, v, w = st["out"]
    if case["kind"] == "batch":
        b = st["batch"]
        dem.dem_batch_run(b.b, case["steps"])
        L = dem.lib()
        for slot, o, n in b.slots:      # the C entry point with device pointers (the binding's reads to the host)
            s = L.dem_batch_get_state(b.b, slot, x.data_ptr() + 24 * o, v.data_ptr() + 24 * o, w.data_ptr() + 24 * o,
                                      dem.DEM_DEVICE)
            if s != dem.DEM_OK:
                raise dem.DemError(s, dem.dem_batch_last_error(b.b))
        return dict(zip("xvw", [x] + _typed(case, (v, w))))
    sim = st["sim"]
    if case["kind"] == "forces":
        dem.dem_set_particles(sim.h, *st["in"])
        dem.dem_get_forces(sim.h, sim.n, v, w)
        return dict(zip("FT", _typed(case, (v, w))))
    out = {}
    if case["kind"] == "until":
        done, disp, _ = dem.dem_run_until(sim.h, case["steps"], 1e-15, 10)
        out = {"steps": done, "disp": np.float32(disp) if case["precision"] == "fp32" else np.float64(disp)}
    else:
        sim.step(case["steps"])
    dem.dem_get_state(sim.h, sim.n, x, v, w)
    out.update(zip("xvw", [x] + _typed(case, (v, w))))
    return out


# -------------------------------------------------------------------------- work
def work(case):
    """Per step: the state of every sphere read and written once (FP32: 56 B in, 48 B out;
    FP64: 80 B in, 76 B out) and every pair's spring read and written once; then the state
    handed out. Operations: about 110 per contact and side (test, law, sums), 60 per sphere."""
    n = case["n"] * case["scenes"]
    if case["kind"] == "batch":
        n = int(n * 0.84)               # mean of the log-uniform sizes
    z = 5.0
    if case["kind"] == "sort":
        return {"bytes": n * (24.0 + 4 + 4) + 4.0 * 1.6 * n, "flops": 12.0 * n}
    f64 = case["precision"] == "fp64"
    spring = 0.0 if case["model"] == "simple" else (z / 2) * 2 * ((24 + 8) if f64 else (12 + 8))
    state = 156.0 if f64 else 104.0
    flops = n * (60.0 + z * (110.0 if case["model"] == "practical" else 70.0))
    if case["kind"] == "forces":
        return {"bytes": n * (76.0 + 48.0), "flops": flops}
    return {"bytes": n * (case["steps"] * (state + spring) + 72.0), "flops": flops * case["steps"]}


# ------------------------------------------------------------------------- exact
def _pairs(x, r, reach):
    """All (i, j), i < j, closer than r_i + r_j + reach, and their sorted keys i n + j."""
    h = 2.0 * float(r.max()) + reach
    lo = x.min(0).values - 0.5 * h
    c = ((x - lo) / h).floor().long()
    d = (c.max(0).values + 2).tolist()
    key = (c[:, 2] * d[1] + c[:, 1]) * d[0] + c[:, 0]
    key, order = torch.sort(key)
    xs, rs = x[order], r[order].double()
    ncell = d[0] * d[1] * d[2]
    start = torch.searchsorted(key, torch.arange(ncell + 1, device=x.device))
    occ = int((start[1:] - start[:-1]).max())
    me = torch.arange(len(r), device=x.device)
    out = []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                off = (dz * d[1] + dy) * d[0] + dx
                if off < 0:
                    continue
                t = (key + off).clamp_(0, ncell - 1)
                ok0 = key + off < ncell
                for s in range(occ):
                    j = start[t] + s
                    ok = ok0 & (j < start[t + 1])
                    if off == 0:
                        ok &= j > me
                    i = me[ok]
                    j = j[ok]
                    near = (xs[j] - xs[i]).square().sum(1) < (rs[i] + rs[j] + reach).square()
                    out.append(torch.stack([i[near], j[near]], 0))
    pr = order[torch.cat(out, 1)]
    i, j = pr.min(0).values, pr.max(0).values
    key = torch.sort(i * len(r) + j).values
    return key // len(r), key % len(r), key


def _dot(a, b):
    return (a * b).sum(1, keepdim=True)


class _Law:
    """Eqs. 1-10 and the optional terms on rows of contacts, in 64 bits."""

    def __init__(self, p):
        self.p = p

    def __call__(self, n, delta, v, rw, Reff, meff, dold, wrel):
        p = self.p
        if p.model == "simple":
            vt = v - n * _dot(v, n)
            return -p.ksp * delta * n - p.kda * v - p.ksh * vt, None, None, None
        vn = n * _dot(v, n)
        vt = v - vn + torch.linalg.cross(rw, n, dim=1)
        d = dold - n * _dot(dold, n) + vt * p.dt
        if p.stiffness == "linear":
            kn = torch.full_like(delta, p.kn)
            kt = torch.full_like(delta, p.kt)
        else:
            s = (delta * Reff).sqrt()
            kn, kt = p.cn * s, p.ct * s
        eta = p.alpha * (kn * meff).sqrt()
        Fn = -kn * delta * n - eta * vn
        if p.terms & 1:
            Fn = torch.where(_dot(Fn, n) > 0, torch.zeros_like(Fn), Fn)
        et = p.alpha_t * (kt * meff).sqrt() if p.terms & 4 else eta
        Ft = -kt * d - et * vt
        fn, ft = Fn.norm(dim=1, keepdim=True), Ft.norm(dim=1, keepdim=True)
        cap = (ft > p.mu * fn) & (ft > 0)
        Fc = Ft * (p.mu * fn / torch.where(ft > 0, ft, torch.ones_like(ft)))
        Ft = torch.where(cap, Fc, Ft)
        d = torch.where(cap & (kt > 0), -(Ft + et * vt) / torch.where(kt > 0, kt, torch.ones_like(kt)), d)
        F = Fn + Ft
        if p.terms & 8:
            F = F + n * (p.k_coh * math.pi * Reff * delta)
        M = None
        if p.terms & 2:
            wn = wrel.norm(dim=1, keepdim=True)
            M = torch.where(wn > 0, -p.mu_roll * Reff * fn * wrel / torch.where(wn > 0, wn, torch.ones_like(wn)),
                            torch.zeros_like(wrel))
        return F, Ft, d, M


def _wall_rows(q, x, r):
    """Contact flag, normal toward the wall, overlap and contact point from p, of every sphere."""
    t = lambda a: torch.tensor(a, dtype=torch.float64, device=x.device).reshape(1, 3)  # noqa: E731
    p, a = t(q["p"]), t(q["n"])
    y = x - p
    if q["kind"] == "plane":
        s = _dot(y, a)
        return r - s, (-a).expand_as(x), y - a * s
    if q["kind"] == "half_plate":
        u = t(q["u"])
        h, s = _dot(y, a), _dot(y, u)
        e = -h * a - torch.where(s < 0, s, torch.zeros_like(s)) * u
        dist = e.norm(dim=1, keepdim=True)
        return r - dist, torch.where(dist > 0, e / dist, (-a).expand_as(x)), y + e
    ax = _dot(y, a)
    rho = y - a * ax
    rr = rho.norm(dim=1, keepdim=True)
    n = rho / torch.where(rr > 0, rr, torch.ones_like(rr))
    return rr + r - q["radius"], n, a * ax + n * q["radius"]


def _exact_run(x, v, w, rf, p, steps, forces=False):
    """`steps` steps (or one force evaluation) in 64 bits; pairs are searched with room to move."""
    r = rf.double()[:, None]
    m = p.rho * 4.0 / 3.0 * math.pi * r ** 3
    I = 0.4 * m * r * r
    reach = 0.3 * R0
    i, j, key = _pairs(x, rf, reach)
    x0 = x
    law = _Law(p)
    dp = torch.zeros((len(i), 3), dtype=torch.float64, device=x.device)
    dw = [torch.zeros_like(x) for _ in p.walls]
    g = torch.tensor(p.g, dtype=torch.float64, device=x.device).reshape(1, 3)
    x, v, w = x.clone(), v.clone(), w.clone()
    disp = torch.zeros((), dtype=torch.float64, device=x.device)
    for _ in range(1 if forces else steps):
        if 2.0 * float((x - x0).norm(dim=1).max()) > 0.8 * reach:
            # some sphere has used up its room: search again, each pair keeps its spring
            i, j, k2 = _pairs(x, rf, reach)
            at = torch.searchsorted(key, k2).clamp_(max=max(len(key) - 1, 0))
            dp = torch.where((key[at] == k2)[:, None], dp[at], torch.zeros_like(dp[:1])) if len(key) else dp[:0]
            key, x0 = k2, x
        F, T = m * g, torch.zeros_like(x)
        e = x[j] - x[i]
        d2 = e.square().sum(1, keepdim=True)
        hit = torch.nonzero((d2 < (r[i] + r[j]).square()).reshape(-1)).reshape(-1)
        a, b = i[hit], j[hit]
        ra, rb = r[a], r[b]
        dist = d2[hit].sqrt()
        n = e[hit] / dist
        f, ft, d, M = law(n, ra + rb - dist, v[a] - v[b], ra * w[a] + rb * w[b], ra * rb / (ra + rb),
                          m[a] * m[b] / (m[a] + m[b]), dp[hit], w[a] - w[b])
        F.index_add_(0, a, f)
        F.index_add_(0, b, -f)
        if ft is not None:
            c = torch.linalg.cross(n, ft, dim=1)
            T.index_add_(0, a, c * ra)
            T.index_add_(0, b, c * rb)
            if M is not None:
                T.index_add_(0, a, M)
                T.index_add_(0, b, -M)
            dp.zero_()
            dp[hit] = d
        for k, q in enumerate(p.walls):
            delta, n, cp = _wall_rows(q, x, r)
            hit = torch.nonzero((delta > 0).reshape(-1)).reshape(-1)
            om = torch.tensor(q["omega"], dtype=torch.float64, device=x.device).reshape(1, 3).expand(len(hit), 3)
            wv = torch.tensor(q["vel"], dtype=torch.float64, device=x.device).reshape(1, 3) + torch.linalg.cross(
                om, cp[hit], dim=1)
            n, rh = n[hit], r[hit]
            f, ft, d, M = law(n, delta[hit], v[hit] - wv, w[hit] * rh, rh, m[hit], dw[k][hit], w[hit] - om)
            F[hit] += f
            if ft is not None:
                T[hit] += torch.linalg.cross(n, ft, dim=1) * rh
                if M is not None:
                    T[hit] += M
                dw[k].zero_()
                dw[k][hit] = d
        if forces:
            return F, T
        v = v + F * (p.dt / m)
        w = w + T * (p.dt / I)
        x = x + v * p.dt
        disp = v.norm(dim=1).max() * p.dt
    return x, v, w, disp


def exact(case, seed):
    if case["kind"] == "sort":
        return None
    if case["kind"] == "batch":
        got = [_exact_run(*s, case["steps"])[:3] for s in _batch_scenes(case, seed)]
        return {k: torch.cat([g[a] for g in got]) for a, k in enumerate("xvw")}
    x, v, w, r, p = _scene(case, seed)
    if case["kind"] == "forces":
        F, T = _exact_run(x, v, w, r, p, 1, forces=True)
        return {"F": F, "T": T}
    x, v, w, disp = _exact_run(x, v, w, r, p, case["steps"])
    out = {"x": x, "v": v, "w": w}
    if case["kind"] == "until":
        out.update(steps=None, disp=float(disp))
    return out
