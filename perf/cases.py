"""The work that a user of this framework has it do, as cases that can be timed and checked.

Every case goes through the public binding (``paper_1606_02862_gb300.pic``): a context is made and
loaded in ``prepare``, ``run`` advances it and reads the results back as a driver script does, into
page-locked host buffers.  A pass goes on from the state that the pass before left, as a run does
between two dumps.  ``exact`` is the same cycle (gather, relativistic Boris push, Esirkepov current,
Yee update) in plain torch at 64 bits.

Kinds of case:
  run       step(n), then E, B and J are read back; with `dump` the particles too (in load order);
            with `monitor` the FP64 diagnostics and the charge density instead of B and J.  The two
            largest read the fields alone, as runs of that size do at most dumps: every particle's
            move of the last step is in J
  batch     independent boxes of different sizes in one context
  window    an open-y laser run: antenna, absorber, particles leaving, a moving window with fresh
            plasma loaded at its top
  restart   a new context from host arrays (a checkpoint), a few steps, and a full dump
"""
import math

import torch

from paper_1606_02862_gb300 import pic

DT = 0.5 / math.sqrt(3.0)  # half the 3D Courant limit for unit cells, as in every workload here
DENS = 0.01                # plasma density of the thermal workloads (and their neutralising background)
PROTON = 1836.15267
LAM, A0, WAIST, DURATION = 32.0, 3.0, 16.0, 40.0  # the laser of the repository's laser workloads
OMEGA = 2.0 * math.pi / LAM
ABSORBER, SIGMA, ANTENNA_Y, RAMP = 32, 1.0, 40, (160, 360)
WINDOW_SLABS = 4           # fresh-plasma slabs a window run keeps in hand
FLOPS = {1: 300.0, 2: 700.0, 3: 1600.0}  # per particle and step, by shape order


def _run(name, nx, ny, nz, ppc, steps, **kw):
    c = dict(name=name, kind="run", nx=nx, ny=ny, nz=nz, ppc=ppc, steps=steps, ions=False, shape=2, energy=False,
             u_th=0.05, dens=DENS, drift=0.0, b0=0.0, foil_lo=0, foil_hi=0, sc="8x4x4", threads=256, plain=False, dump=False,
             monitor=False)
    c.update(kw)
    return c


def listed():
    return [
        # one step of the smallest workload with its fields looked at after it: launches and latency
        _run("step_cic_32", 32, 32, 32, 2, 1, shape=1, u_th=0.01, b0=0.1, sc="4x4x4", threads=128),
        # the usual loop of a small study: some steps, then the time-series diagnostics and rho
        _run("monitor_tsc_64", 64, 64, 64, 8, 10, monitor=True, dump=True),
        # an ordinary run in a box that no large supercell divides, energy-conserving gather, particle dump
        _run("run_cic_ragged", 92, 132, 100, 8, 30, shape=1, energy=True, sc="4x4x4", threads=128, dump=True),
        # the cubic shape, for low-noise runs
        _run("run_pcs_96", 96, 96, 96, 8, 12, shape=3, dump=True),
        # shear flow of electrons and ions at 16 particles per cell each, 128^3: the evaluation size
        _run("shear_128", 128, 128, 128, 16, 20, ions=True, u_th=0.005, drift=0.2),
        # the headline box: 256^3, 134 million particles
        _run("thermal_256", 256, 256, 256, 8, 20),
        # a dense foil in a large vacuum box: field update and empty supercells beside a few full ones
        _run("foil_192", 192, 768, 192, 16, 20, ions=True, u_th=0.02, dens=0.3, foil_lo=352, foil_hi=372),
        # fields alone (a vacuum box: antenna and cavity studies, the field solver's own runs)
        _run("vacuum_256", 256, 256, 256, 0, 100),
        # the FP64 form, taken to check a result in full precision
        _run("plain_tsc_64", 64, 64, 64, 8, 4, plain=True, dump=True),
        # a parameter scan: many small boxes of uneven size and filling in one context
        dict(name="batch_uneven", kind="batch", boxes=24, lo=16, hi=96, max_ppc=16, steps=20, pick=3),
        # laser run with a moving window
        dict(name="window_64", kind="window", nx=64, ny=512, nz=64, ppc=4, steps=14, shifts=2),
        # restart from a checkpoint and dump a new one
        _run("restart_128", 128, 128, 128, 8, 4, kind="restart", dump=True),
    ]


def _edge(rng, lo, hi, of):
    return max(lo, of * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / of))


def draw(rng):
    """One more case of the ranges of listed(): box edges from 16 to 256 (multiples of 4), up to 30
    million particles, from one step to a few dozen, every shape, gather, supercell and form."""
    kind = rng.choice(["run"] * 8 + ["plain", "vacuum", "batch", "window", "restart", "monitor"])
    if kind == "batch":
        return dict(kind="batch", boxes=rng.randint(4, 32), lo=16, hi=rng.choice([48, 64, 80]),
                    max_ppc=rng.randint(4, 16), steps=rng.randint(2, 24), pick=rng.randrange(1 << 20))
    if kind == "window":
        return dict(kind="window", nx=8 * rng.randint(3, 10), ny=8 * rng.randint(30, 60), nz=4 * rng.randint(6, 18),
                    ppc=rng.randint(1, 4), steps=14, shifts=rng.randint(1, 3))
    sc, threads = rng.choice([("8x4x4", 256)] * 4 + [("4x4x4", 128)] * 3 + [("8x8x4", 256), ("8x8x8", 256), ("8x4x4", 128),
                                                   ("4x4x4", 256), ("4x4x4", 64)])
    shape = rng.choice([1, 2, 2, 2, 3])
    if shape == 3:
        sc, threads = rng.choice([("8x4x4", 256), ("4x4x4", 128)])
    of = [int(v) for v in sc.split("x")]
    ppc = rng.choice([1, 2, 3, 4, 6, 8, 8, 12, 16, 24])
    most = 2.0e6 if kind == "plain" else 3.0e7
    n = [_edge(rng, 16, 200, a) for a in of]
    if kind == "vacuum":
        return _run("", *(_edge(rng, 32, 256, a) for a in of), 0, rng.randint(4, 60), sc=sc, threads=threads) | {"name": ""}
    ions = rng.random() < 0.35
    while n[0] * n[1] * n[2] * ppc * (2 if ions else 1) > most:
        a = n.index(max(n))
        n[a] -= of[a]
    steps = rng.randint(1, 4) if kind == "plain" else max(1, round(math.exp(rng.uniform(0.0, math.log(40.0)))))
    c = _run("", *n, ppc, steps, ions=ions, shape=min(shape, 2) if kind == "plain" else shape,
             energy=rng.random() < 0.3, u_th=round(rng.uniform(0.005, 0.1), 4), sc=sc, threads=threads,
             drift=rng.choice([0.0, 0.0, 0.2]), b0=rng.choice([0.0, 0.1]), dump=rng.random() < 0.4,
             plain=kind == "plain", monitor=kind == "monitor")
    if kind == "restart":
        c["kind"] = "restart"
        c["steps"] = min(steps, 6)
    c.pop("name")
    return c


# ------------------------------------------------------------------ inputs

def _rng(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _species(c):
    out = [(-1.0, 1.0)]
    if c.get("ions"):
        out.append((1.0, PROTON))
    return out


def _plasma(g, n3, ppc, u_th, drift, y_lo, y_hi, lo=0, hi=None, dens=DENS, weight=None):
    """Particles [lo, hi) of a plasma of ppc uniform positions in every cell of the rows y_lo <= y <
    y_hi, cell after cell, Maxwellian momenta about +-drift along x (two shear slabs); x, u, w."""
    nx, ny, nz = n3
    rows = y_hi - y_lo
    hi = nx * rows * nz * ppc if hi is None else hi
    cell = torch.arange(lo, hi, device="cuda", dtype=torch.int64).div_(ppc, rounding_mode="floor")
    x = torch.rand((hi - lo, 3), generator=g, device="cuda", dtype=torch.float64)
    x[:, 0] += cell % nx
    x[:, 1] += cell.div(nx, rounding_mode="floor") % rows + y_lo
    x[:, 2] += cell.div(nx * rows, rounding_mode="floor")
    x.clamp_(max=max(n3) * (1.0 - 2.0 ** -52))
    u = torch.randn((hi - lo, 3), generator=g, device="cuda", dtype=torch.float64) * u_th
    if drift:
        up = (x[:, 1] >= ny / 4) & (x[:, 1] < 3 * ny / 4)
        u[:, 0] += torch.where(up, 1.0, -1.0) * (drift / math.sqrt(1.0 - drift * drift))
    if weight is None:
        w = torch.full((hi - lo,), dens / ppc, device="cuda", dtype=torch.float64)
    else:
        w = weight(torch.floor(x[:, 1]) + 0.5) / ppc
    return x, u, w


def _rows(c):
    return (c["foil_lo"], c["foil_hi"]) if c.get("foil_hi") else (0, c["ny"])


def _count(c):
    lo, hi = _rows(c)
    return c["nx"] * (hi - lo) * c["nz"] * c["ppc"]


def _pieces(c, seed, most=1 << 23):
    """The particles of a run case in pieces, as (species, x, u, w) on the device, always the same for a seed."""
    n, (lo, hi) = _count(c), _rows(c)
    for s, (_, m) in enumerate(_species(c)):
        g = _rng(seed * 7919 + s)
        for b in range(0, n, most):
            yield (s, *_plasma(g, (c["nx"], c["ny"], c["nz"]), c["ppc"], c["u_th"] / math.sqrt(m), c["drift"], lo, hi, b, min(n, b + most),
                             c["dens"]))


def _fields0(c, seed):
    """E and B at the start: a uniform B_z; a vacuum box and a foil run start from random fields
    (every mode present), a restart from those of a developed plasma's size."""
    f = torch.zeros((2, 3, c["nz"], c["ny"], c["nx"]), device="cuda", dtype=torch.float64)
    if c["b0"]:
        f[1, 2] = c["b0"]
    if c["ppc"] == 0 or c["foil_hi"] or c["kind"] == "restart":
        f += 0.01 * torch.randn(f.shape, generator=_rng(seed * 7919 + 11), device="cuda", dtype=torch.float64)
    return f


def _pinned(*shape, dtype=torch.float64):
    return torch.empty(shape, dtype=dtype, pin_memory=True)


def _host(t):
    return _pinned(*t.shape, dtype=t.dtype).copy_(t)


def _load(ctx, box, s, x, u, w):
    x, u, w = _host(x), _host(u), _host(w)
    ctx.load_particles_ptr(box, s, x.shape[0], x.data_ptr(), u.data_ptr(), w.data_ptr())


def _context(c, grids, **kw):
    kinds = [pic.Species(q, m, c["shape"], True, pic.GATHER_ENERGY if c["energy"] else pic.GATHER_MOMENTUM)
             for q, m in _species(c)]
    return pic.Context(grids, (1.0, 1.0, 1.0), DT, kinds,
                       precision=pic.PRECISION_FP64_PLAIN if c["plain"] else pic.PRECISION_MIXED,
                       sc=tuple(int(v) for v in c["sc"].split("x")), threads_per_sc=c["threads"],
                       track_ids=c["dump"], **kw)


def _batch_boxes(c):
    """Edge, ppc and u_th of the boxes of a batch case: the same for every seed."""
    g = torch.Generator().manual_seed(c["pick"])
    out = []
    for _ in range(c["boxes"]):
        r = torch.rand(3, generator=g, dtype=torch.float64).tolist()
        edge = c["lo"] + 8 * int(r[0] * ((c["hi"] - c["lo"]) // 8 + 1))
        out.append((edge, 1 + int(r[1] * c["max_ppc"]), 0.01 + 0.09 * r[2]))
    return out


def _batch_box(c, b, seed):
    edge, ppc, u_th = _batch_boxes(c)[b]
    return _plasma(_rng(seed * 7919 + b), (edge,) * 3, ppc, u_th, 0.0, 0, edge)


def _density(row):
    n0 = 0.01 * OMEGA ** 2
    return n0 * ((row - RAMP[0]) / (RAMP[1] - RAMP[0])).clamp(0.0, 1.0)


def _window_plasma(c, seed):
    """Electrons and protons of a window run, and its fresh slabs (4 rows each, for the window's top)."""
    n3, first, slabs = (c["nx"], c["ny"], c["nz"]), [], []
    lo = min(RAMP[0], c["ny"] - 4)
    for s, m in enumerate((1.0, PROTON)):
        first.append(_plasma(_rng(seed * 7919 + s), n3, c["ppc"], 0.001 / math.sqrt(m), 0.0, lo, c["ny"], weight=_density))
    for k in range(WINDOW_SLABS):
        slabs.append([_plasma(_rng(seed * 7919 + 101 + 2 * k + s), n3, c["ppc"], 0.001 / math.sqrt(m), 0.0, c["ny"] - 4, c["ny"],
                              weight=lambda row: torch.full_like(row, 0.01 * OMEGA ** 2)) for s, m in enumerate((1.0, PROTON))])
    return first, slabs


# ------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    c = dict(case)
    st = {"case": c}
    if c["kind"] == "batch":
        boxes = _batch_boxes(c)
        ctx = pic.Context([(e, e, e) for e, _, _ in boxes], (1.0, 1.0, 1.0), DT, [pic.Species(-1.0, 1.0, 2)],
                          sc=(8, 4, 4), threads_per_sc=256)
        for b in range(len(boxes)):
            ctx.set_background(b, DENS)
            _load(ctx, b, 0, *_batch_box(c, b, seed))
        sizes = [3 * e ** 3 for e, _, _ in boxes]
        st.update(ctx=ctx, sizes=sizes, E=_pinned(sum(sizes)), B=_pinned(sum(sizes)), J=_pinned(sum(sizes)))
    elif c["kind"] == "window":
        ctx = pic.Context([(c["nx"], c["ny"], c["nz"])], (1.0, 1.0, 1.0), DT,
                          [pic.Species(-1.0, 1.0, 2), pic.Species(1.0, PROTON, 2)], sc=(8, 4, 4), threads_per_sc=256)
        ctx.set_boundary(0, open_y=True, absorber_cells=ABSORBER, absorber_sigma=SIGMA)
        ctx.set_antenna(0, **_antenna(c))
        first, slabs = _window_plasma(c, seed)
        for s in range(2):
            _load(ctx, 0, s, *first[s])
        st.update(ctx=ctx, slabs=[[tuple(_host(t) for t in p) for p in k] for k in slabs], at=0)
        st.update({f: _pinned(3, c["nz"], c["ny"], c["nx"]) for f in "EBJ"})
    else:
        n, kinds = _count(c), len(_species(c))
        st.update({f: _pinned(3, c["nz"], c["ny"], c["nx"]) for f in "EBJ"})
        if c["dump"]:
            st["x"], st["u"], st["id"] = _pinned(n, 3), _pinned(n, 3), _pinned(n, dtype=torch.int64)
            st["x0"] = [torch.empty((n, 3), device="cuda", dtype=torch.float64) for _ in range(kinds)]
        if c["kind"] == "restart":
            st["load"] = [tuple(_pinned(n, k) for k in (3, 3)) + (_pinned(n),) for _ in range(kinds)]
        else:
            st["ctx"] = _context(c, [(c["nx"], c["ny"], c["nz"])])
            if kinds == 1:
                st["ctx"].set_background(0, DENS)
        at = [0] * kinds
        for s, x, u, w in _pieces(c, seed):
            m = slice(at[s], at[s] + x.shape[0])
            at[s] += x.shape[0]
            if c["dump"]:
                st["x0"][s][m] = x
            if c["kind"] == "restart":
                for to, t in zip(st["load"][s], (x, u, w)):
                    to[m].copy_(t)
            else:
                _load(st["ctx"], 0, s, x, u, w)
        f = _fields0(c, seed).cpu()
        if c["kind"] == "restart":
            st["f0"] = (f[0].clone(), f[1].clone())
        elif f.any():
            st["ctx"].write_fields(0, pic.FIELD_E, f[0])
            st["ctx"].write_fields(0, pic.FIELD_B, f[1])
    torch.cuda.synchronize()
    return st


def _antenna(c):
    return dict(plane_y=ANTENNA_Y, E0=A0 * OMEGA, omega=OMEGA, w0=WAIST, xc=c["nx"] / 2.0, zc=c["nz"] / 2.0, tau=DURATION,
                t0=2.0 * DURATION)


def _read_fields(ctx, st, fields="EBJ"):
    out = {}
    for f in fields:
        ctx.read_fields_ptr(0, {"E": pic.FIELD_E, "B": pic.FIELD_B, "J": pic.FIELD_J}[f], st[f].data_ptr())
        out[f] = st[f]
    return out


def _read_particles(ctx, st):
    """Displacement since the load (nearest image, so that the seam is no jump) and momentum of every
    particle, in load order."""
    c, out = st["case"], {}
    edges = torch.tensor([c["nx"], c["ny"], c["nz"]], device="cuda", dtype=torch.float64)
    for s, x0 in enumerate(st["x0"]):
        ctx.read_particles_ptr(0, s, x0.shape[0], st["x"].data_ptr(), st["u"].data_ptr(), None, st["id"].data_ptr())
        order = st["id"].cuda()
        x, u = torch.empty_like(x0), torch.empty_like(x0)
        x[order] = st["x"].cuda()
        u[order] = st["u"].cuda()
        out["moved%d" % s], out["u%d" % s] = _nearest(x - x0, edges), u
    return out


def _nearest(dx, edges):
    return dx - edges * torch.round(dx / edges)


def run(state):
    st, c = state, state["case"]
    if c["kind"] == "batch":
        ctx = st["ctx"]
        ctx.step(c["steps"])
        for f, which in (("E", pic.FIELD_E), ("B", pic.FIELD_B), ("J", pic.FIELD_J)):
            at = st[f].data_ptr()
            for b, n in enumerate(st["sizes"]):
                ctx.read_fields_ptr(b, which, at)
                at += 8 * n
        return {"E": st["E"], "B": st["B"], "J": st["J"]}
    if c["kind"] == "window":
        ctx = st["ctx"]
        for _ in range(c["shifts"]):
            ctx.step(c["steps"])
            ctx.shift_window(0, 4)
            for s, (x, u, w) in enumerate(st["slabs"][st["at"] % WINDOW_SLABS]):
                ctx.load_particles_ptr(0, s, x.shape[0], x.data_ptr(), u.data_ptr(), w.data_ptr())
            st["at"] += 1
        ctx.step(c["steps"])
        return _read_fields(ctx, st)
    if c["kind"] == "restart":
        with _context(c, [(c["nx"], c["ny"], c["nz"])]) as ctx:
            for s, (x, u, w) in enumerate(st["load"]):
                ctx.load_particles_ptr(0, s, x.shape[0], x.data_ptr(), u.data_ptr(), w.data_ptr())
            ctx.write_fields(0, pic.FIELD_E, st["f0"][0])
            ctx.write_fields(0, pic.FIELD_B, st["f0"][1])
            ctx.step(c["steps"])
            return {**_read_fields(ctx, st), **(_read_particles(ctx, st) if c["dump"] else {})}
    ctx = st["ctx"]
    ctx.step(c["steps"])
    if c["monitor"]:
        out = {**_read_fields(ctx, st, "E"), "diagnostics": ctx.diagnostics(0), "rho": ctx.read_fields(0, pic.FIELD_RHO)}
    else:
        out = _read_fields(ctx, st)
    return {**out, **(_read_particles(ctx, st) if c["dump"] else {})}


# ------------------------------------------------------------------ work and tolerance

def _sizes(c):
    """(cells, particles, steps, fields read, particles dumped or loaded) of a pass."""
    if c["kind"] == "batch":
        b = _batch_boxes(c)
        return sum(e ** 3 for e, _, _ in b), sum(e ** 3 * p for e, p, _ in b), c["steps"], 3, 0
    if c["kind"] == "window":
        cells = c["nx"] * c["ny"] * c["nz"]
        full = 2 * c["ppc"] * c["nx"] * c["nz"]
        return cells, full * max(4, c["ny"] - RAMP[0]), c["steps"] * (c["shifts"] + 1), 3, 4 * full * c["shifts"]
    n = _count(c) * len(_species(c))
    return c["nx"] * c["ny"] * c["nz"], n, c["steps"], 2 if c["monitor"] else 3, n * (int(c["dump"]) + (c["kind"] == "restart"))


def work(case):
    """Bytes: per step 32 B read and 28 B written per particle, per cell E, B read and J written by the
    push (36 B) and E, B, J read, E, B written by the field update (60 B); twice that in the FP64 form;
    and the FP64 host values of what is read back or loaded with their 32-bit originals."""
    cells, n, steps, fields, moved = _sizes(case)
    wide = 2 if case.get("plain") else 1
    per_cell = 96 if n else 60
    return {"bytes": wide * steps * (60.0 * n + per_cell * cells) + 36.0 * cells * fields + 88.0 * moved,
            "flops": steps * (FLOPS[case.get("shape", 2)] * n + 54.0 * cells)}


def tolerance(case):
    """About four times what two runs of one build, and the FP64 cycle below, differ by: the mixed form
    5e-6 (FP32 fields, momenta and offsets; the current rounds in fixed point and adds up in any
    order) and 5e-5 at the worst value; the FP64 form 6e-15 and 1e-13."""
    return {"rel": 5e-14, "max": 2e-12} if case.get("plain") else {"rel": 2e-5, "max": 4e-4}


# ------------------------------------------------------------------ the same in 64 bits

def _S(order, d):
    a = d.abs()
    if order == 0:
        return torch.ones_like(a)  # nearest node: the only one in its window
    if order == 1:
        return (1.0 - a).clamp(min=0.0)
    if order == 2:
        t = (1.5 - a).clamp(min=0.0)
        return torch.where(a <= 0.5, 0.75 - a * a, 0.5 * t * t)
    t = (2.0 - a).clamp(min=0.0)
    return torch.where(a < 1.0, (4.0 - 6.0 * a * a + 3.0 * a * a * a) / 6.0, t * t * t / 6.0)


class _Box64:
    """One box in FP64 on the device.  F: (3, nz, ny, nx); particles [x, u, w] per species."""

    def __init__(self, n3, species, order, energy, E=None, B=None, open_y=None):
        self.n, self.species, self.order, self.energy, self.open_y, self.steps = n3, species, order, energy, open_y, 0
        shape = (3, n3[2], n3[1], n3[0])
        self.E = torch.zeros(shape, device="cuda", dtype=torch.float64) if E is None else E.clone()
        self.B = torch.zeros_like(self.E) if B is None else B.clone()
        self.J = torch.zeros_like(self.E)
        self.parts = [None] * len(species)

    def _axis(self, x, axis, stagger, order):
        """Node indices (wrapped) and weights along one axis."""
        xs = x[:, axis] - stagger
        b = torch.floor(xs - 0.5 * (order - 1))
        return [((b + k).long() % self.n[axis], _S(order, xs - (b + k))) for k in range(order + 1)]

    def _gather(self, x):
        nx, ny, _ = self.n
        half = self.order - 1 if self.energy else self.order
        ax = [[self._axis(x, a, 0.0, self.order), self._axis(x, a, 0.5, half)] for a in range(3)]
        out = []
        for F, sides in ((self.E, ((1, 0, 0), (0, 1, 0), (0, 0, 1))), (self.B, ((0, 1, 1), (1, 0, 1), (1, 1, 0)))):
            for comp, (sx, sy, sz) in enumerate(sides):
                f = F[comp].reshape(-1)
                acc = torch.zeros_like(x[:, 0])
                for iz, wz in ax[2][sz]:
                    for iy, wy in ax[1][sy]:
                        row, wzy = (iz * ny + iy) * nx, wz * wy
                        for ix, wx in ax[0][sx]:
                            acc.addcmul_(f[row + ix], wzy * wx)
                out.append(acc)
        return torch.stack(out[:3], 1), torch.stack(out[3:], 1)

    def _push(self, s, x, u, w):
        q, m = self.species[s]
        E, B = self._gather(x)
        eps = q * DT / (2.0 * m)
        um = u + eps * E
        t = eps * B / torch.sqrt(1.0 + (um * um).sum(1, keepdim=True))
        up = um + torch.linalg.cross(um, t)
        u = um + torch.linalg.cross(up, 2.0 * t / (1.0 + (t * t).sum(1, keepdim=True))) + eps * E
        x1 = x + DT * u / torch.sqrt(1.0 + (u * u).sum(1, keepdim=True))
        idx, S0, DS = [], [], []
        for a in range(3):
            b = torch.floor(torch.minimum(x[:, a], x1[:, a]) - 0.5 * (self.order - 1))
            nodes = [b + k for k in range(self.order + 2)]
            idx.append([v.long() % self.n[a] for v in nodes])
            S0.append([_S(self.order, x[:, a] - v) for v in nodes])
            DS.append([_S(self.order, x1[:, a] - v) - s0 for v, s0 in zip(nodes, S0[a])])
        stride = (1, self.n[0], self.n[0] * self.n[1])
        cf = -q * w / DT
        for d in range(3):
            e, f = (d + 1) % 3, (d + 2) % 3
            flat = self.J[d].reshape(-1)
            P = [cf * DS[d][0]]
            for k in range(1, self.order + 1):
                P.append(P[-1] + cf * DS[d][k])
            for i in range(self.order + 2):
                for j in range(self.order + 2):
                    T = S0[e][i] * (S0[f][j] + 0.5 * DS[f][j]) + DS[e][i] * (0.5 * S0[f][j] + DS[f][j] / 3.0)
                    at = idx[e][i] * stride[e] + idx[f][j] * stride[f]
                    for k in range(self.order + 1):
                        flat.index_add_(0, at + idx[d][k] * stride[d], P[k] * T)
        return x1, u

    def _half_b(self):
        E = self.E
        d = lambda c, axis: torch.roll(E[c], -1, 2 - axis) - E[c]  # noqa: E731
        self.B[0] -= 0.5 * DT * (d(2, 1) - d(1, 2))
        self.B[1] -= 0.5 * DT * (d(0, 2) - d(2, 0))
        self.B[2] -= 0.5 * DT * (d(1, 0) - d(0, 1))

    def _full_e(self):
        B = self.B
        d = lambda c, axis: B[c] - torch.roll(B[c], 1, 2 - axis)  # noqa: E731
        self.E[0] += DT * (d(2, 1) - d(1, 2) - self.J[0])
        self.E[1] += DT * (d(0, 2) - d(2, 0) - self.J[1])
        self.E[2] += DT * (d(1, 0) - d(0, 1) - self.J[2])

    def step(self, count, piece=1 << 21):
        edges = torch.tensor(self.n, device="cuda", dtype=torch.float64)
        for _ in range(count):
            self.J.zero_()
            for s, p in enumerate(self.parts):
                if p is None:
                    continue
                for b in range(0, p[0].shape[0], piece):
                    m = slice(b, b + piece)
                    p[0][m], p[1][m] = self._push(s, p[0][m], p[1][m], p[2][m])
                if self.open_y:
                    keep = (p[0][:, 1] >= 0.0) & (p[0][:, 1] < self.n[1])
                    p[:] = [t[keep] for t in p]
                p[0] -= edges * torch.floor(p[0] / edges)
            if self.open_y:
                self._antenna()
            self._half_b()
            self._full_e()
            self._half_b()
            if self.open_y:
                self._absorb()
            self.steps += 1

    def _antenna(self):
        a = self.open_y
        kappa = 2.0 * math.asin(math.sin(0.5 * a["omega"] * DT) / DT)
        t = (self.steps + 0.5) * DT - a["t0"]
        now = -2.0 * a["E0"] * math.cos(0.5 * kappa) * math.exp(-(t / a["tau"]) ** 2) * math.cos(a["omega"] * t)
        x = torch.arange(self.n[0], device="cuda", dtype=torch.float64) + 0.5 - a["xc"]
        z = torch.arange(self.n[2], device="cuda", dtype=torch.float64)[:, None] - a["zc"]
        self.J[0, :, a["plane_y"], :] += now * torch.exp(-(x * x + z * z) / a["w0"] ** 2)

    def _absorb(self):
        y = torch.arange(self.n[1], device="cuda", dtype=torch.float64)

        def factor(y):
            depth = torch.maximum(ABSORBER - y, y - (self.n[1] - ABSORBER)).div(ABSORBER).clamp(0.0, 1.0)
            return torch.exp(-SIGMA * depth * depth)[:, None]

        whole, half = factor(y), factor(y + 0.5)
        for c, (fe, fb) in enumerate(((whole, half), (half, whole), (whole, half))):
            self.E[c] *= fe
            self.B[c] *= fb

    def shift(self, cells):
        for F in (self.E, self.B):
            F[:, :, :-cells] = F[:, :, cells:].clone()
            F[:, :, -cells:] = 0.0
        for p in self.parts:
            p[0][:, 1] -= cells
            p[:] = [t[p[0][:, 1] >= 0.0] for t in p]

    def rho(self, background):
        nx, ny, nz = self.n
        out = torch.full((nz * ny * nx,), background, device="cuda", dtype=torch.float64)
        for (q, _), p in zip(self.species, self.parts):
            ax = [self._axis(p[0], a, 0.0, self.order) for a in range(3)]
            for iz, wz in ax[2]:
                for iy, wy in ax[1]:
                    for ix, wx in ax[0]:
                        out.index_add_(0, (iz * ny + iy) * nx + ix, q * p[2] * wz * wy * wx)
        return out.view(nz, ny, nx)

    def diagnostics(self, background):
        rho = self.rho(background)
        div = sum(self.E[a] - torch.roll(self.E[a], 1, 2 - a) for a in range(3))
        kin = sum(float((p[2] * m * (p[1] * p[1]).sum(1) / (torch.sqrt(1.0 + (p[1] * p[1]).sum(1)) + 1.0)).sum())
                  for (_, m), p in zip(self.species, self.parts))
        field = 0.5 * float((self.E * self.E).sum() + (self.B * self.B).sum())
        return torch.tensor([field, kin, float(rho.sum()), float((div - rho).abs().max())], dtype=torch.float64), rho


def exact(case, seed):
    c = dict(case)
    cells, n, steps, _, _ = _sizes(c)
    if (n * (3.0 if c.get("shape") == 3 else 1.0) + 0.1 * cells) * steps > 6e8:
        return None  # minutes in plain torch; the smaller cases cover the same code
    if c["kind"] == "batch":
        got = []
        for b, (edge, _, _) in enumerate(_batch_boxes(c)):
            box = _Box64((edge,) * 3, [(-1.0, 1.0)], 2, False)
            box.parts[0] = list(_batch_box(c, b, seed))
            box.step(c["steps"])
            got.append([t.reshape(-1) for t in (box.E, box.B, box.J)])
        return {f: torch.cat([g[k] for g in got]) for k, f in enumerate("EBJ")}
    if c["kind"] == "window":
        box = _Box64((c["nx"], c["ny"], c["nz"]), [(-1.0, 1.0), (1.0, PROTON)], 2, False, open_y=_antenna(c))
        first, slabs = _window_plasma(c, seed)
        box.parts = [list(p) for p in first]
        for k in range(c["shifts"]):
            box.step(c["steps"])
            box.shift(4)
            box.parts = [[torch.cat(t) for t in zip(p, new)] for p, new in zip(box.parts, slabs[k % WINDOW_SLABS])]
        box.step(c["steps"])
        return {"E": box.E, "B": box.B, "J": box.J}
    f = _fields0(c, seed)
    box = _Box64((c["nx"], c["ny"], c["nz"]), _species(c), c["shape"], c["energy"], f[0], f[1])
    for s in range(len(_species(c)) if n else 0):
        box.parts[s] = [torch.cat(t) for t in zip(*((x, u, w) for k, x, u, w in _pieces(c, seed) if k == s))]
    first = [p[0].clone() for p in box.parts if p is not None] if c["dump"] else []
    box.step(c["steps"])
    if c["monitor"]:
        diag, rho = box.diagnostics(DENS if len(_species(c)) == 1 else 0.0)
        out = {"E": box.E, "diagnostics": diag, "rho": rho}
    else:
        out = {"E": box.E, "B": box.B, "J": box.J}
    edges = torch.tensor(box.n, device="cuda", dtype=torch.float64)
    for s, x0 in enumerate(first):
        out["moved%d" % s], out["u%d" % s] = _nearest(box.parts[s][0] - x0, edges), box.parts[s][1]
    return out
