"""Performance cases of the implicit PIC library: short runs through its public entry points.

A "run" pass is what a user's program does with one set of inputs: it empties
the handle, sets the initial fields, loads the species (arrays in device
memory), advances the steps and reads the state back (moments, fields,
energies, counts; in the FP64 form the particles too, as a checkpoint does).
The collision and ionisation cases call the pass after every step, as a run
with these processes does; the serving case submits a burst of independent
runs to a server and collects their results.  The FP32 form's grids are
handed on as FP32 tensors on the device, the precision they have (its particle
order is not returned: a last-bit change of a position may move a particle to
the next cell).

exact() repeats a pass in plain FP64 torch: cell and offset per particle, one
scatter-add per corner, 3x3 solves by cofactors, the time-centred field system
by BiCGSTAB to 1e-14.
"""
import ctypes
import math
import random

import numpy as np
import torch

from paper_1308_2590_gb300 import pic
from paper_1308_2590_gb300 import workloads as W

DEV = "cuda"
LAM = 2.0 * math.pi
MP = 1836.0                                  # proton mass (m_e)
CARBON_IP = (11.2603, 24.3833)               # eV, C0 -> C1+, C1+ -> C2+
LN_LAMBDA = 10.0
KAPPA = LAM * 2.8179403262e-15 / 0.8e-6      # r_e omega / c of a 0.8 um laser
OMEGA0 = LAM * 299792458.0 / 0.8e-6
FIELD_AU = 9.1093837015e-31 * 299792458.0 * OMEGA0 / 1.602176634e-19 / 5.14220674763e11
TIME_AU = (1.0 / OMEGA0) / 2.4188843265857e-17
HARTREE_EV = 27.211386245988
LASER_TAU = 30e-15 * OMEGA0
STEP_SEED = 20240607                         # seed of the collision and ionisation draws


def _run(name, box, nx, ny, ppc, steps, **kw):
    c = dict(name=name, kind="run", box=box, nx=nx, ny=ny, ppc=ppc, steps=steps, precision="fp64", field="literal",
             shape=1, exact_deposit=False, tile=8, x0=0, thick=nx, density=1.0, a0=0.0, particles=False)
    c.update(kw)
    return c


def listed():
    return [
        # the small plain run: 64 x 64 periodic plasma, 131,072 particles, 50 time-centred steps; launches,
        # grid barriers and host latency count
        _run("uniform-64-cn", "uniform", 64, 64, 16, 50, field="cn", tile=16, particles=True),
        # one small run of a served parameter scan on its own handle (ragged last tile row), FP32
        _run("scan-192x317-fp32", "foil", 192, 317, 20, 60, precision="fp32", x0=86, thick=19, density=80.0, a0=8.0),
        # the particle-dominated laser foil in both forms (6.55M particles)
        _run("foil-1024x512", "foil", 1024, 512, 64, 8, x0=150, thick=100, density=100.0, a0=5.0, particles=True),
        _run("foil-1024x512-fp32", "foil", 1024, 512, 64, 24, precision="fp32", x0=150, thick=100, density=100.0,
             a0=5.0),
        # the field-dominated laser foil (8.4M nodes, 0.33M particles)
        _run("thin-foil-4096x2048", "foil", 4096, 2048, 4, 16, x0=150, thick=20, density=50.0, a0=5.0,
             particles=True),
        # the largest: hot periodic plasma, 67M particles, time-centred solve, FP32
        _run("uniform-1024-cn-fp32", "uniform", 1024, 1024, 32, 4, field="cn", precision="fp32", tile=16),
        # higher-order shapes on the foil: quadratic in FP64, cubic in FP32
        _run("foil-quadratic", "foil", 1024, 512, 64, 4, shape=2, x0=150, thick=100, density=100.0, a0=5.0,
             particles=True),
        _run("foil-cubic-fp32", "foil", 1024, 512, 64, 6, shape=3, precision="fp32", x0=150, thick=100,
             density=100.0, a0=5.0),
        # the foil with the time-centred solve and absorbing walls, exact (reproducible) deposit
        _run("foil-cn-walls", "foil", 1024, 512, 32, 4, field="cn", exact_deposit=True, x0=150, thick=100,
             density=100.0, a0=5.0, particles=True),
        # a collisional foil: e-e, e-i, i-i passes after every step
        _run("foil-collisions", "foil", 1024, 512, 32, 3, kind="collide", x0=150, thick=100, density=100.0, a0=5.0,
             particles=True),
        # an ionising carbon foil: the field-ionisation pass after every step (grids and counts per species come
        # back: how many particles a species has differs from input to input)
        _run("carbon-ionisation", "carbon", 1024, 512, 16, 6, kind="ionize", x0=150, thick=100, density=100.0,
             a0=5.0),
        # a burst of small independent FP32 runs on one server
        dict(name="serve-burst", kind="serve", runs=12, nmax=256, ppcmax=24, steps=40, mix=7),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["uniform", "foil", "foil", "shape", "walls", "collide", "ionize", "serve"])
    if kind == "serve":
        return dict(kind="serve", runs=rng.randint(2, 12), nmax=rng.choice([96, 128, 192, 256]),
                    ppcmax=rng.randint(6, 24), steps=rng.randint(10, 40), mix=rng.randint(8, 10 ** 6))
    prec = rng.choice(["fp64", "fp32"])
    if kind == "uniform":
        nx, ny = rng.choice([32, 64, 96, 128, 192, 256, 512]), rng.choice([32, 64, 90, 128, 256, 512])
        c = _run("", "uniform", nx, ny, _logint(rng, 4, 40), rng.randint(2, 12), field="cn", precision=prec,
                 tile=rng.choice([8, 16]))
    else:
        nx, ny = _logint(rng, 96, 1200), _logint(rng, 64, 700)
        thick = max(6, nx // rng.randint(8, 14))
        c = _run("", "foil", nx, ny, _logint(rng, 4, 72), rng.randint(2, 6), precision=prec,
                 x0=min(150, (nx - thick) // 2), thick=thick, density=rng.uniform(10.0, 150.0),
                 a0=rng.uniform(1.0, 12.0), exact_deposit=rng.random() < 0.25)
        if kind == "shape":
            c.update(shape=rng.choice([2, 3, 4]), steps=rng.randint(2, 4))
        elif kind == "walls":
            c.update(field="cn", ppc=_logint(rng, 4, 32))
        elif kind == "collide":
            c.update(kind="collide", precision="fp64", ppc=_logint(rng, 3, 40), steps=2)
        elif kind == "ionize":
            c.update(kind="ionize", box="carbon", precision="fp64", ppc=_logint(rng, 4, 20))
    c["particles"] = c["precision"] == "fp64" and c["kind"] != "ionize"
    del c["name"]
    return c


# ---------------------------------------------------------------- what a case means (no library code)

def _phys(c):
    """Cell size, time step, species (q, m, weight, thermal u) and laser of a run case."""
    if c["box"] == "uniform":
        dx, dt, tau = 0.02, 0.5, 0.0
        sp = [(-1.0, 1.0, 1.0), (1.0, MP, 1.0)]
    else:
        dx, dt, tau = LAM / 40.0, 0.01 * LAM, LASER_TAU
        sp = [(-1.0, 1.0, c["density"]), (1.0, 1836.15267343, c["density"])]
        if c["box"] == "carbon":
            n = c["density"] / 6.0
            sp = [(-1.0, 1.0, n)] + [(float(z), 12.0 * MP, n) for z in range(3)]
    w = [n * dx * dx / c["ppc"] for _, _, n in sp]
    uth = [math.sqrt(1.0 / (510.99895 * m)) for _, m, _ in sp]
    return dict(dx=dx, dt=dt, tau=tau, periodic=c["box"] == "uniform", sp=[(q, m) for q, m, _ in sp], w=w, uth=uth)


def _particles(c, seed):
    """Initial particles of every species (FP64 tensors on the device): uniform in the slab's cells, cell by
    cell, Maxwellian momenta; the species share positions.  A carbon foil starts as electrons, C0 and C1+,
    with no C2+."""
    p = _phys(c)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    ppc, ncx = c["ppc"], c["thick"]
    n = ppc * ncx * c["ny"]
    k = torch.arange(n, device=DEV, dtype=torch.int64) // ppc
    rnd = lambda: torch.rand(n, generator=gen, device=DEV, dtype=torch.float64).clamp_(max=1.0 - 1e-9)  # noqa: E731
    x = ((c["x0"] + k % ncx).double() + rnd()) * p["dx"]
    y = ((k // ncx).double() + rnd()) * p["dx"]
    del k
    out = []
    for s in range(len(p["sp"])):
        if c["box"] == "carbon" and s == 3:
            out.append(None)
            continue
        u = [torch.randn(n, generator=gen, device=DEV, dtype=torch.float64) * p["uth"][s] for _ in range(3)]
        out.append([x, y] + u + [torch.full((n,), p["w"][s], device=DEV, dtype=torch.float64)])
    return out


def _initial_fields(c, seed):
    """Smooth initial E (nodes) and H (cells): a few plane waves along each axis, as of a run in progress."""
    rng = np.random.default_rng([int(seed), 77])
    nxn = c["nx"] if _phys(c)["periodic"] else c["nx"] + 1
    amp = 0.06 if c["box"] == "foil" else 0.01
    i, j = np.arange(nxn) / c["nx"], np.arange(c["ny"]) / c["ny"]
    out = []
    for n in (nxn, c["nx"]):
        f = np.zeros((3, c["ny"], n))
        for comp in range(3):
            for _ in range(2):
                a, b = rng.integers(1, 5), rng.integers(1, 4)
                px, py = rng.uniform(0, LAM, 2)
                f[comp] += amp * rng.uniform(0.5, 1.0) * np.outer(np.sin(LAM * b * j + py), np.sin(LAM * a * i[:n] + px))
        out.append(f)
    return out


def _serve_runs(c):
    """The run cases of a serving burst: foils of different sizes, densities and laser strengths."""
    r = random.Random(c["mix"])
    out = []
    for _ in range(c["runs"]):
        nx, ny = 64 * r.randint(1, c["nmax"] // 64), 32 * r.randint(2, c["nmax"] // 32)
        thick = max(1, int(round(nx / 10)))
        out.append(_run("", "foil", nx, ny, r.randint(4, c["ppcmax"]), c["steps"], precision="fp32",
                        x0=min(150, (nx - thick) // 2), thick=thick, density=r.uniform(10.0, 200.0),
                        a0=r.uniform(1.0, 20.0)))
    return out


# ---------------------------------------------------------------- the library's side

def _config(c):
    p = _phys(c)
    return W.RunConfig(
        name="case", nx=c["nx"], ny=c["ny"], dx=p["dx"], dy=p["dx"], dt=p["dt"], steps=c["steps"],
        bc_x=W.BC_PERIODIC if p["periodic"] else W.BC_ABSORBING,
        field_mode=W.FIELD_CN if c["field"] == "cn" else W.FIELD_LITERAL,
        precision=W.PREC_FP32 if c["precision"] == "fp32" else W.PREC_FP64,
        deposit=W.DEPOSIT_DETERMINISTIC if c["exact_deposit"] else W.DEPOSIT_ATOMIC,
        species=[W.Species(q, m, c["ppc"], 1.0, 1.0) for q, m in p["sp"]],
        laser=W.Laser(a0=c["a0"], omega=1.0, tau=p["tau"], t0=p["tau"], pol=0), tile_nx=c["tile"], tile_ny=c["tile"],
        shape=c["shape"])


def _pinned(*shape, dtype=torch.float64):
    return torch.empty(shape, dtype=dtype, pin_memory=True).numpy()


def _check(rc, what):
    if rc != pic.PIC_OK:
        raise RuntimeError("%s: %s" % (what, pic.lib().pic_last_error().decode()))


def prepare(case, seed):
    if case["kind"] == "serve":
        subs = []
        for k, c in enumerate(_serve_runs(case)):
            parts = []
            for a in _particles(c, seed * 1000 + k):
                host = _pinned(6, a[0].numel())
                host[...] = torch.stack(a).cpu().numpy()
                parts.append(dict(zip(("x", "y", "ux", "uy", "uz", "w"), host)))
            subs.append((_config(c), parts))
        return dict(case=case, server=pic.Server(mem_budget=8 << 30), subs=subs)
    c, cfg = case, _config(case)
    nxn = c["nx"] if cfg.bc_x == W.BC_PERIODIC else c["nx"] + 1
    data = _particles(c, seed)
    n = [0 if a is None else a[0].numel() for a in data]
    room = list(n)
    if c["kind"] == "ionize":
        room = [(4 if s == 0 else 2) * max(n) for s in range(len(n))]   # each ion may give two electrons
    sd = (pic.PicSpeciesData * len(data))()
    for s, a in enumerate(data):
        sd[s].n = n[s]
        if a is not None:
            sd[s].x, sd[s].y, sd[s].ux, sd[s].uy, sd[s].uz, sd[s].w = [v.data_ptr() for v in a]
    E0, H0 = _pinned(3, c["ny"], nxn), _pinned(3, c["ny"], c["nx"])
    E0[...], H0[...] = _initial_fields(c, seed)
    out = dict(E=_pinned(3, c["ny"], nxn), H=_pinned(3, c["ny"], c["nx"]))
    if c["nx"] * c["ny"] <= 1 << 21:   # (a field-dominated run is read for its fields)
        out["moments"] = _pinned(13, c["ny"], nxn)
    if c["particles"]:
        out["particles"] = [(_pinned(m, dtype=torch.int32), _pinned(6, m)) for m in room]
    return dict(case=case, g=pic.Pic(cfg, capacity=room), data=data, sd=sd, E0=E0, H0=H0, out=out)


def _ptr(a):
    return ctypes.c_void_p(a.ctypes.data)


def _read(st):
    """The state after the steps: moments, fields, energies, counts and (where asked) the particles."""
    g, c, out, L = st["g"], st["case"], st["out"], pic.lib()
    res = {}
    if "moments" in out:
        res["moments"] = g.pic_moments(out["moments"])
    _check(L.pic_fields(g.h, _ptr(out["E"]), _ptr(out["H"])), "pic_fields")
    res["E"], res["H"] = out["E"], out["H"]
    if c["precision"] == "fp32":
        for k in res:
            res[k] = torch.from_numpy(res[k]).to(DEV, non_blocking=True).float()
    d = g.pic_diagnostics()
    res["kinetic"], res["count"] = d["kinetic"], d["count"]
    if c["kind"] == "ionize":
        res["counts"] = [g.pic_particle_count(s) for s in range(g.nsp)]
    if "particles" in out:
        res["particles"] = []
        for s, (cell, val) in enumerate(out["particles"]):
            n = g.pic_particle_count(s)
            v = [val[k, :n] for k in range(6)]
            _check(L.pic_save_particles(g.h, s, _ptr(cell), *[_ptr(a) for a in v]), "pic_save_particles")
            res["particles"].append([cell[:n]] + v)
    return res


def run(state):
    c = state["case"]
    if c["kind"] == "serve":
        srv = state["server"]
        ids = [srv.submit(cfg, parts, c["steps"], keep_grids=True) for cfg, parts in state["subs"]]
        srv.wait_all(120.0)
        res = []
        for rid in ids:
            d, (M, E, H) = srv.result(rid, grids=True)
            srv.release(rid)
            res.append([torch.from_numpy(a).float() for a in (M, E, H)] + [d["kinetic"], d["count"]])
        return res
    g = state["g"]
    g.pic_clear_particles()
    g.pic_set_fields(state["E0"], state["H0"])
    g.pic_set_step(0)
    _check(pic.lib().pic_load_species(g.h, len(state["data"]), state["sd"]), "pic_load_species")
    if c["kind"] == "run":
        g.pic_step(c["steps"])
        return _read(state)
    done = []
    for k in range(c["steps"]):
        g.pic_step(1)
        if c["kind"] == "collide":
            done.append(g.pic_collide([(0, 0), (0, 1), (1, 1)], seed=STEP_SEED, ln_lambda=LN_LAMBDA, kappa=KAPPA))
        else:
            done.append(g.pic_ionize([(1, 2, 0, CARBON_IP[0]), (2, 3, 0, CARBON_IP[1])], seed=STEP_SEED,
                                     field_unit_au=FIELD_AU, time_unit_au=TIME_AU))
    res = _read(state)
    res["events"] = done
    return res


def work(case):
    """Bytes and operations a pass cannot do without: the loads (FP64 arrays read, state written), per step
    every particle's state read and its changed part written and the grid planes of the field solve, and the
    state read back."""
    if case["kind"] == "serve":
        w = [work(c) for c in _serve_runs(case)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    c = case
    rs = 4 if c["precision"] == "fp32" else 8
    n = {"uniform": 2, "foil": 2, "carbon": 3}[c["box"]] * c["ppc"] * c["thick"] * c["ny"]
    nodes = c["nx"] * c["ny"]
    per = 4 + 6 * rs + 4 + 5 * rs
    b = n * (48 + 4 + 6 * rs) + c["steps"] * (n * per + nodes * 30 * rs)
    b += nodes * 8 * (6 + 6 + (13 if nodes <= 1 << 21 else 0)) + (n * 52 if c["particles"] else 0)
    f = c["steps"] * (n * (98 + 38 * (c["shape"] + 1) ** 2) + nodes * 60)
    if c["kind"] == "collide":
        b += c["steps"] * n * 3 * 7 * rs
        f += c["steps"] * n * 300
    if c["kind"] == "ionize":
        b += c["steps"] * n * (4 + 2 * rs)
        f += c["steps"] * n * 100
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- the same pass in plain FP64 torch

CHUNK = 1 << 21


def _bspline(n, x):
    a = x.abs()
    if n == 2:
        return torch.where(a <= 0.5, 0.75 - a * a, 0.5 * (1.5 - a).clamp(min=0) ** 2)
    if n == 3:
        return torch.where(a <= 1, 2.0 / 3.0 - a * a + 0.5 * a ** 3, (2 - a).clamp(min=0) ** 3 / 6.0)
    mid = (55 + 20 * a - 120 * a ** 2 + 80 * a ** 3 - 16 * a ** 4) / 96.0
    return torch.where(a <= 0.5, 115.0 / 192.0 - 0.625 * a * a + 0.25 * a ** 4,
                       torch.where(a <= 1.5, mid, (5 - 2 * a).clamp(min=0) ** 4 / 384.0))


def _axis(order, c, f, n, periodic):
    """Node indices and weights along one axis."""
    if order == 1:
        nodes = [(c, 1.0 - f), (c + 1, f)]
    else:
        first = c - (order - 1) // 2 if order % 2 else c - order // 2 + (f >= 0.5).long()
        nodes = [(first + k, _bspline(order, (first + k - c).double() - f)) for k in range(order + 1)]
    return [(i % n if periodic else i.clamp(0, n), w) for i, w in nodes]


class _Sim:
    def __init__(self, c, seed, fields=True):
        self.c, p = c, _phys(c)
        self.nx, self.ny, self.per = c["nx"], c["ny"], p["periodic"]
        self.nxn = self.nx if self.per else self.nx + 1
        self.h, self.dt, self.sp, self.tau = p["dx"], p["dt"], p["sp"], p["tau"]
        if fields:
            E, H = [torch.from_numpy(f).to(DEV) for f in _initial_fields(c, seed)]
        else:
            E = torch.zeros(3, self.ny, self.nxn, dtype=torch.float64, device=DEV)
            H = torch.zeros(3, self.ny, self.nx, dtype=torch.float64, device=DEV)
        self.E, self.H, self.step = E, H, 0
        self.P = []
        for a in _particles(c, seed):
            if a is None:
                z = torch.zeros(0, dtype=torch.float64, device=DEV)
                self.P.append([z.long(), z.long()] + [z] * 6)
                continue
            sx, sy = a[0] / self.h, a[1] / self.h
            cx, cy = sx.floor(), sy.floor()
            self.P.append([cx.long(), cy.long(), sx - cx, sy - cy] + a[2:])
        for s in range(len(self.P)):
            self.sort(s)
        self.B = self.node_average(self.H)
        self.deposit()

    # order: tiles, cells in a tile, stayers before arrivals
    def keys(self, s):
        t, (cx, cy) = self.c["tile"], self.P[s][:2]
        tx, ty = min(t, self.nx), min(t, self.ny)
        ntx = -(-self.nx // tx)
        tile = (cy // ty) * ntx + cx // tx
        return tile, tile * (tx * ty) + (cy % ty) * tx + cx % tx

    def sort(self, s, old_tile=None):
        tile, key = self.keys(s)
        key = 2 * key + (0 if old_tile is None else (tile != old_tile).long())
        order = torch.sort(key, stable=True)[1]
        self.P[s] = [a[order] for a in self.P[s]]

    def node_average(self, H):
        s = H + H.roll(1, 1)
        if self.per:
            return 0.25 * (s + s.roll(1, 2))
        B = torch.empty(3, self.ny, self.nxn, dtype=H.dtype, device=DEV)
        B[:, :, 1:-1] = 0.25 * (s[:, :, 1:] + s[:, :, :-1])
        B[:, :, 0], B[:, :, -1] = 0.5 * s[:, :, 0], 0.5 * s[:, :, -1]
        return B

    def curl_h(self, H):
        dy = (H - H.roll(1, 1)) / self.h          # between cell rows
        ay = 0.5 * (H + H.roll(1, 1))
        out = torch.zeros(3, self.ny, self.nxn, dtype=H.dtype, device=DEV)
        if self.per:
            ddy, ddx = 0.5 * (dy + dy.roll(1, 2)), (ay - ay.roll(1, 2)) / self.h
            out[0], out[1], out[2] = ddy[2], -ddx[2], ddx[1] - ddy[0]
            return out
        ddy, ddx = 0.5 * (dy[:, :, 1:] + dy[:, :, :-1]), (ay[:, :, 1:] - ay[:, :, :-1]) / self.h
        out[0, :, 1:-1], out[1, :, 1:-1], out[2, :, 1:-1] = ddy[2], -ddx[2], ddx[1] - ddy[0]
        for e in (0, -1):
            out[0, :, e], out[2, :, e] = dy[2, :, e], -dy[0, :, e]
        return out

    def curl_e(self, E):
        dy, ay = (E.roll(-1, 1) - E) / self.h, 0.5 * (E.roll(-1, 1) + E)
        if self.per:
            ddy, ddx = 0.5 * (dy + dy.roll(-1, 2)), (ay.roll(-1, 2) - ay) / self.h
        else:
            ddy, ddx = 0.5 * (dy[:, :, 1:] + dy[:, :, :-1]), (ay[:, :, 1:] - ay[:, :, :-1]) / self.h
        return torch.stack([ddy[2], -ddx[2], ddx[1] - ddy[0]])

    def nodes(self, cx, cy, fx, fy, order):
        ax = _axis(order, cx, fx, self.nx, self.per)
        ay = _axis(order, cy, fy, self.ny, True)
        return [(j * self.nxn + i, wx * wy) for j, wy in ay for i, wx in ax]

    def gather(self, F, nodes):
        rows = F.reshape(3, -1).t().contiguous() if F.shape[0] == 3 else F
        out = 0.0
        for i, w in nodes:
            out = out + w[:, None] * rows[i]
        return out.unbind(1)

    @staticmethod
    def rot(b, v):
        vb = v[0] * b[0] + v[1] * b[1] + v[2] * b[2]
        den = 1.0 + b[0] ** 2 + b[1] ** 2 + b[2] ** 2
        return [(v[k] + v[(k + 1) % 3] * b[(k + 2) % 3] - v[(k + 2) % 3] * b[(k + 1) % 3] + vb * b[k]) / den
                for k in range(3)]

    def deposit(self):
        M = torch.zeros(self.ny * self.nxn, 13, dtype=torch.float64, device=DEV)
        Brow = self.B.reshape(3, -1).t().contiguous()
        for (q, m), P in zip(self.sp, self.P):
            for o in range(0, P[0].numel(), CHUNK):
                cx, cy, fx, fy, ux, uy, uz, w = [a[o:o + CHUNK] for a in P]
                nodes = self.nodes(cx, cy, fx, fy, self.c["shape"])
                ig = 1.0 / torch.sqrt(1.0 + ux * ux + uy * uy + uz * uz)
                b = [q * self.dt / (2.0 * m) * ig * v for v in self.gather(Brow, nodes)]
                one, zero = torch.ones_like(ux), torch.zeros_like(ux)
                cols = [self.rot(b, [one if r == k else zero for r in range(3)]) for k in range(3)]
                cs = w * q * q * self.dt ** 2 / (4.0 * m) * ig
                dj = self.rot(b, [ux, uy, uz])
                val = torch.stack([w * q] + [cs * cols[k][r] for r in range(3) for k in range(3)] +
                                  [w * q * ig * d for d in dj], 1)
                for i, wt in nodes:
                    M.index_add_(0, i, wt[:, None] * val)
        M = M.t().reshape(13, self.ny, self.nxn) / (self.h * self.h)
        if not self.per:
            M[:, :, 0] *= 2.0
            M[:, :, -1] *= 2.0
        self.M = M

    def laser(self, t):
        a0 = self.c["a0"]
        if t < 0 or a0 == 0:
            return 0.0
        env = math.exp(-2.0 * math.log(2.0) * (t - self.tau) ** 2 / self.tau ** 2) if self.tau > 0 else 1.0
        return a0 * math.sin(t) * env

    @staticmethod
    def cofactor_solve(A, r):
        """z of A z = r, A[row][col] and r planes."""
        cof = [[A[(i + 1) % 3][(j + 1) % 3] * A[(i + 2) % 3][(j + 2) % 3] -
                A[(i + 1) % 3][(j + 2) % 3] * A[(i + 2) % 3][(j + 1) % 3] for j in range(3)] for i in range(3)]
        det = A[0][0] * cof[0][0] + A[0][1] * cof[0][1] + A[0][2] * cof[0][2]
        return torch.stack([(cof[0][k] * r[0] + cof[1][k] * r[1] + cof[2][k] * r[2]) / det for k in range(3)])

    def IS(self, sign=1.0):
        return [[sign * self.M[1 + 3 * r + k] + (1.0 if r == k else 0.0) for k in range(3)] for r in range(3)]

    def field_literal(self, t1):
        dt, h, E, t0 = self.dt, self.h, self.E, t1 - self.dt
        ch, A, Bm = self.curl_h(self.H), self.IS(), self.IS(-1.0)
        r = [sum(Bm[k][j] * E[j] for j in range(3)) + dt * (ch[k] - self.M[10 + k]) for k in range(3)]
        N = self.cofactor_solve(A, r)
        if not self.per:
            kap = (dt - h) / (dt + h)
            for w, v in ((0, 1), (-1, -2)):
                N[0, :, w] = E[0, :, w] + dt * ch[0, :, w]
                for comp in (1, 2):
                    inc = [self.laser(t) if (w == 0 and comp == 1) else 0.0 for t in (t1, t0, t1 - h, t0 - h)]
                    N[comp, :, w] = inc[0] + (E[comp, :, v] - inc[3]) + kap * ((N[comp, :, v] - inc[2]) -
                                                                              (E[comp, :, w] - inc[1]))
        return 0.5 * (E + N), N, self.H - dt * self.curl_e(N)

    def field_cn(self, t1):
        dt, h, E, t0 = self.dt, self.h, self.E, t1 - self.dt
        A3 = self.IS()
        S = self.M[1:10].clone()
        dj = self.M[10:13].clone()
        cw, cv = 1.0 / dt + 1.0 / h, 1.0 / dt - 1.0 / h
        if not self.per:
            S[:, :, 0] = S[:, :, -1] = 0.0
            dj[:, :, 0] = dj[:, :, -1] = 0.0
            for r in range(3):
                for k in range(3):
                    A3[r][k][:, 0] = A3[r][k][:, -1] = 1.0 if r == k else 0.0

        def op(X):
            Y = X + 0.25 * dt * dt * self.curl_h(self.curl_e(X))
            Y += torch.stack([S[3 * r] * X[0] + S[3 * r + 1] * X[1] + S[3 * r + 2] * X[2] for r in range(3)])
            if not self.per:
                for w, v in ((0, 1), (-1, -2)):
                    Y[1:, :, w] = X[1:, :, w] + cv / cw * X[1:, :, v]
            return Y

        b = E + 0.5 * dt * (self.curl_h(self.H) - dj)
        if not self.per:
            for w, v in ((0, 1), (-1, -2)):
                b[1:, :, w] = (E[1:, :, w] + E[1:, :, v]) / (dt * cw)
            f = [self.laser(t) for t in (t0, t1, t0 - h, t1 - h)]
            b[1, :, 0] += (-(f[0] + f[2]) / dt + cw * 0.5 * (f[0] + f[1]) + cv * 0.5 * (f[2] + f[3])) / cw
        if self.per:
            ex = torch.exp(1j * LAM * torch.arange(self.nx, device=DEV, dtype=torch.float64) / self.nx)[None, :]
            ey = torch.exp(1j * LAM * torch.arange(self.ny, device=DEV, dtype=torch.float64) / self.ny)[:, None]
            Dx, Dy = (ex - 1) / h * (1 + ey) / 2, (ey - 1) / h * (1 + ex) / 2
            z = torch.zeros_like(Dx)
            curl = lambda a, c: torch.stack([z, z, c, z, z, -a, -c, a, z], -1).reshape(*z.shape, 3, 3)  # noqa: E731
            sym = curl(-Dx.conj(), -Dy.conj()) @ curl(Dx, Dy)
            mean = torch.eye(3, device=DEV, dtype=torch.float64) + S.mean((1, 2)).reshape(3, 3)
            inv = torch.linalg.inv(mean + 0.25 * dt * dt * sym)
            pre = lambda r: torch.fft.ifft2(torch.einsum("yxab,byx->ayx", inv, torch.fft.fft2(r))).real  # noqa: E731
        else:
            pre = lambda r: self.cofactor_solve(A3, r)  # noqa: E731
        dot = lambda a, c: float((a * c).sum())  # noqa: E731
        X, nb = pre(b), math.sqrt(dot(b, b)) + 1e-300
        for _ in range(12):   # BiCGSTAB, restarted from the true residual
            r = b - op(X)
            if math.sqrt(dot(r, r)) < 1e-15 * nb:
                break
            r0, p, rho, n0 = r.clone(), r.clone(), dot(r, r), math.sqrt(dot(r, r))
            for _ in range(60):
                ph = pre(p)
                v = op(ph)
                al = rho / dot(r0, v)
                s = r - al * v
                sh = pre(s)
                t = op(sh)
                om = dot(t, s) / max(dot(t, t), 1e-300)
                X = X + al * ph + om * sh
                r = s - om * t
                if math.sqrt(dot(r, r)) < 1e-4 * n0:
                    break
                rho1 = dot(r0, r)
                p = r + (rho1 / rho) * (al / om) * (p - om * v)
                rho = rho1
        return X, 2.0 * X - E, self.H - dt * self.curl_e(X)

    def advance(self):
        t1 = (self.step + 1) * self.dt
        X, N, H = self.field_literal(t1) if self.c["field"] == "literal" else self.field_cn(t1)
        Erow, Brow = [F.reshape(3, -1).t().contiguous() for F in (X, self.B)]
        for s, (q, m) in enumerate(self.sp):
            P, k, new = self.P[s], q * self.dt / (2.0 * m), []
            tile = self.keys(s)[0]
            for o in range(0, P[0].numel(), CHUNK):
                cx, cy, fx, fy, ux, uy, uz, w = [a[o:o + CHUNK] for a in P]
                nodes = self.nodes(cx, cy, fx, fy, self.c["shape"])
                E, B = self.gather(Erow, nodes), self.gather(Brow, nodes)
                ig = 1.0 / torch.sqrt(1.0 + ux * ux + uy * uy + uz * uz)
                ub = self.rot([k * v * ig for v in B], [ux + k * E[0], uy + k * E[1], uz + k * E[2]])
                sx, sy = fx + self.dt / self.h * ub[0] * ig, fy + self.dt / self.h * ub[1] * ig
                nx, ny = cx + sx.floor().long(), (cy + sy.floor().long()) % self.ny
                if self.per:
                    nx = nx % self.nx
                new.append([nx, ny, sx - sx.floor(), sy - sy.floor(), 2 * ub[0] - ux, 2 * ub[1] - uy, 2 * ub[2] - uz, w])
            if not new:
                continue
            P = [torch.cat(a) for a in zip(*new)]
            if not self.per:
                live = (P[0] >= 0) & (P[0] < self.nx)
                if not bool(live.all()):
                    P, tile = [a[live] for a in P], tile[live]
            self.P[s] = P
            self.sort(s, tile)
        self.E, self.H = N, H
        self.B = self.node_average(H)
        self.deposit()
        self.step += 1

    def collide(self, entries):
        pairs = 0
        for k, (sa, sb) in enumerate(entries):
            ca = self.P[sa][1] * self.nx + self.P[sa][0]
            cell, cnt = torch.unique_consecutive(ca, return_counts=True)
            first = torch.cumsum(cnt, 0) - cnt
            run = torch.repeat_interleave(torch.arange(cell.numel(), device=DEV), cnt)
            pos = torch.arange(ca.numel(), device=DEV) - first[run]
            wa = torch.zeros(cell.numel(), dtype=torch.float64, device=DEV).index_add_(0, run, self.P[sa][7])
            if sa == sb:
                n, nL = cnt[run], (wa / self.h ** 2)[run]
                odd = (n % 2 == 1) & (n >= 3)
                base = torch.arange(ca.numel(), device=DEV)
                stages = [(((n % 2 == 0) & (pos % 2 == 0)) | (odd & (pos >= 3) & (pos % 2 == 1)), 1, False),
                          (odd & (pos == 0), 1, True), (odd & (pos == 1), 1, True), (odd & (pos == 2), -2, True)]
                for mask, off, half in stages:
                    i = base[mask]
                    self.scatter(sa, i, sa, i + off, nL[i], k, half)
                    pairs += i.numel()
                continue
            cb = self.P[sb][1] * self.nx + self.P[sb][0]
            cellb, cntb = torch.unique_consecutive(cb, return_counts=True)
            firstb = torch.cumsum(cntb, 0) - cntb
            runb = torch.repeat_interleave(torch.arange(cellb.numel(), device=DEV), cntb)
            wb = torch.zeros(cellb.numel(), dtype=torch.float64, device=DEV).index_add_(0, runb, self.P[sb][7])
            table = torch.full((self.nx * self.ny,), -1, dtype=torch.int64, device=DEV)
            table[cellb] = torch.arange(cellb.numel(), device=DEV)
            both = table[cell] >= 0
            fa, na, wa, rb = first[both], cnt[both], wa[both], table[cell[both]]
            fb, nb, wb = firstb[rb], cntb[rb], wb[rb]
            nL = torch.minimum(wa, wb) / self.h ** 2
            for s1, f1, n1, s2, f2, n2, sel in ((sa, fa, na, sb, fb, nb, na >= nb), (sb, fb, nb, sa, fa, na, na < nb)):
                f1, n1, f2, n2, l = f1[sel], n1[sel], f2[sel], n2[sel], nL[sel]
                r = 0
                while f1.numel():   # round r: each particle of the smaller species once
                    m = torch.minimum(n2, n1 - r * n2)
                    keep = m > 0
                    f1, n1, f2, n2, l, m = f1[keep], n1[keep], f2[keep], n2[keep], l[keep], m[keep]
                    if not f1.numel():
                        break
                    rep = torch.repeat_interleave(torch.arange(m.numel(), device=DEV), m)
                    j = torch.arange(rep.numel(), device=DEV) - (torch.cumsum(m, 0) - m)[rep]
                    self.scatter(s1, (f1 + r * n2)[rep] + j, s2, f2[rep] + j, l[rep], k, False)
                    pairs += rep.numel()
                    r += 1
        self.deposit()
        return pairs

    def scatter(self, s1, i, s2, j, nL, entry, half):
        (q1, m1), (q2, m2) = self.sp[s1], self.sp[s2]
        u1, u2 = [self.P[s1][4 + k][i] for k in range(3)], [self.P[s2][4 + k][j] for k in range(3)]
        w1, w2 = self.P[s1][7][i], self.P[s2][7][j]
        v = [((x >> 11) & ((1 << 53) - 1)).double() * 2.0 ** -53 for x in _philox(i, 16 + entry, self.step, 1)]
        g = [a - b for a, b in zip(u1, u2)]
        gm = torch.sqrt(g[0] ** 2 + g[1] ** 2 + g[2] ** 2)
        mu = m1 * m2 / (m1 + m2)
        var = q1 * q1 * q2 * q2 * nL * LN_LAMBDA * KAPPA * self.dt / (2.0 * mu * mu * gm ** 3) * (0.5 if half else 1.0)
        de = torch.sqrt(var) * torch.sqrt(-2.0 * torch.log(1.0 - v[0])) * torch.cos(LAM * v[1])
        sT, cT = 2.0 * de / (1.0 + de * de), 2.0 * de * de / (1.0 + de * de)
        gp, cp, sp = torch.sqrt(g[0] ** 2 + g[1] ** 2), torch.cos(LAM * v[2]), torch.sin(LAM * v[2])
        dg = [g[0] / gp * g[2] * sT * cp - g[1] / gp * gm * sT * sp - g[0] * cT,
              g[1] / gp * g[2] * sT * cp + g[0] / gp * gm * sT * sp - g[1] * cT, -gp * sT * cp - g[2] * cT]
        ok, wm = gm > 0, torch.maximum(w1, w2)
        a1, a2 = (ok & (v[3] < w2 / wm)), (ok & (v[3] < w1 / wm))
        for k in range(3):
            self.P[s1][4 + k][i] = torch.where(a1, u1[k] + m2 / (m1 + m2) * dg[k], u1[k])
            self.P[s2][4 + k][j] = torch.where(a2, u2[k] - m1 / (m1 + m2) * dg[k], u2[k])

    def ionize(self, chains):
        moved = []
        for a, t, e, ip_ev in chains:
            P = self.P[a]
            F = self.gather(self.E, self.nodes(P[0], P[1], P[2], P[3], 1))
            F = torch.sqrt(F[0] ** 2 + F[1] ** 2 + F[2] ** 2) * FIELD_AU
            ip, Z = ip_ev / HARTREE_EV, self.sp[t][0]
            n, K = Z / math.sqrt(2.0 * ip), 2.0 * (2.0 * ip) ** 1.5
            Fp = F.clamp(max=K / (3.0 * (2.0 * n - 1.0)) if n > 0.5 else math.inf)
            rate = 2.0 ** (2.0 * n) / (n * math.gamma(2.0 * n)) * ip * (K / Fp) ** (2.0 * n - 1.0) * torch.exp(-K / (3.0 * Fp))
            prob = torch.where(F > 0, -torch.expm1(-rate * self.dt * TIME_AU), 0.0)
            x = _philox(torch.arange(F.numel(), device=DEV), a, self.step, 0)[0]
            go = ((x >> 11) & ((1 << 53) - 1)).double() * 2.0 ** -53 < prob
            moved.append((t, e, [v[go] for v in P], go))
        for (a, _, _, _), (_, _, _, go) in zip(chains, moved):
            self.P[a] = [v[~go] for v in self.P[a]]
        for t, e, m, _ in moved:
            for s in (t, e):
                self.P[s] = [torch.cat([x, y]) for x, y in zip(self.P[s], m)]
        for s in {s for t, e, _, _ in moved for s in (t, e)}:
            self.sort(s)
        self.deposit()
        return sum(int(go.sum()) for _, _, _, go in moved)

    def kinetic(self):
        return sum(float((P[7] * m * (torch.sqrt(1.0 + P[4] ** 2 + P[5] ** 2 + P[6] ** 2) - 1.0)).sum())
                   for (_, m), P in zip(self.sp, self.P))


def _philox(index, c1, c2, c3):
    """Philox-4x64-10 (Salmon et al., SC 2011) at counter (index, c1, c2, c3), key (STEP_SEED, 0); int64 words."""
    lo32 = 0xFFFFFFFF
    signed = lambda v: v - (1 << 64) if v >> 63 else v  # noqa: E731

    def mulhilo(a, b):
        al, ah = a & lo32, a >> 32
        bl, bh = b & lo32, (b >> 32) & lo32
        ll, lh, hl, hh = bl * al, bh * al, bl * ah, bh * ah
        hi32 = lambda v: (v >> 32) & lo32  # noqa: E731
        mid = hi32(ll) + (lh & lo32) + (hl & lo32)
        return hh + hi32(lh) + hi32(hl) + (mid >> 32), b * signed(a)

    x = [index.clone()] + [torch.full_like(index, v) for v in (c1, c2, c3)]
    k0, k1 = STEP_SEED, 0
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B97F4A7C15) % (1 << 64), (k1 + 0xBB67AE8584CAA73B) % (1 << 64)
        h0, l0 = mulhilo(0xD2E7470EE14C6C93, x[0])
        h1, l1 = mulhilo(0xCA5A826395121157, x[2])
        x = [h1 ^ x[1] ^ signed(k0), l1, h0 ^ x[3] ^ signed(k1), l0]
    return x


def exact(case, seed):
    if case["kind"] == "serve":
        out = []
        for k, c in enumerate(_serve_runs(case)):
            sim = _Sim(c, seed * 1000 + k, fields=False)
            for _ in range(c["steps"]):
                sim.advance()
            out.append([v.cpu() for v in (sim.M, sim.E, sim.H)] + [sim.kinetic(), None])
        return out
    sim = _Sim(case, seed)
    for _ in range(case["steps"]):
        sim.advance()
        if case["kind"] == "collide":
            sim.collide([(0, 0), (0, 1), (1, 1)])
        elif case["kind"] == "ionize":
            sim.ionize([(1, 2, 0, CARBON_IP[0]), (2, 3, 0, CARBON_IP[1])])
    res = dict(E=sim.E.cpu(), H=sim.H.cpu(), kinetic=sim.kinetic(), count=None)
    if case["nx"] * case["ny"] <= 1 << 21:
        res["moments"] = sim.M.cpu()
    if case["particles"]:
        res["particles"] = [[None] + [v.cpu() for v in P[2:]] for P in sim.P]
    if case["kind"] != "run":
        res["events"] = [None] * case["steps"]
    return res
