"""The work this solver is used for, as cases that can be timed and checked.

A case is a dict of plain values.  `prepare` makes what a user's program holds before the call
(grids with their fields placed, batches, particles, buffers for the results), `run` advances it
by the case's steps through the public bindings and hands back the whole state and the recorded
energies (a scan: every instance's energies and axion field, what a scan is run for), and `exact`
computes the same state in 64 bits with plain torch, from the scheme of arXiv 2406.16796 Sec.
2.2-2.4 written out on whole arrays.

Outputs are grouped by order, since components that vanish by symmetry hold only rounding noise:
order0 (E0 and B0), order1 (E1 and B1), phi (phi^{n+1/2}) and second (phi^{n-1/2} in FP64, the
increment phi^{n+1/2} - phi^{n-1/2} in FP32).  FP64 grids are read to pinned host memory at
integer time; FP32 grids are packed on the device, where the single-pass kernels keep E half a
step ahead.  The energies H_phi, H_g0, H_g1 are those of the diagnostics ring.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2406_16796_gb300 import axp, batch, group
from paper_2406_16796_gb300.workloads import AxionSpec, GridSpec, LaserSpec

K0 = 2.0 * math.pi  # the laser's wave number: lengths are in its wavelength


# ---- the cases ----

def listed():
    return [
        # the 1D conversion run: CW wave, uniform B, periodic box, energies recorded as it goes
        dict(name="conversion_1d", kind="line", nx=4096, bc="periodic", precision="fp64", m=0.0, steps=2000, every=100),
        # a short 1D pulse that leaves through absorbing edges: the smallest call, one launch's latency per step
        dict(name="pulse_1d_absorbing", kind="line", nx=2048, bc="pml", precision="fp32", m=0.5, steps=192, every=0),
        # the parameter scan: 512 uneven 1D runs advanced together
        dict(name="scan_512", kind="scan", count=512, steps=512),
        # 2D laser pulse through B along z, absorbing on every side, at the size it is quoted on
        dict(name="pulse_2d", kind="pulse", nx=4096, ny=2048, pol="z", axion_bc="pml", precision="fp64", m=0.5,
             window=0, steps=100, every=100),
        # the same in FP32 split, in a window that follows the pulse
        dict(name="pulse_2d_window", kind="pulse", nx=4096, ny=2048, pol="z", axion_bc="pml", precision="fp32", m=0.5,
             window=64, steps=400, every=100),
        # the boundary benchmark: an axion pulse leaving a 400 x 400 box, no laser
        dict(name="boundary_2d", kind="axion2d", nx=400, ny=400, axion_bc="pml", precision="fp64", m=6.5e-4, steps=100,
             every=0),
        # 2D pulse with the outflow condition on the axion
        dict(name="outflow_2d", kind="pulse", nx=1024, ny=512, pol="z", axion_bc="outflow", precision="fp64", m=0.0,
             window=0, steps=100, every=100),
        # 2D pulse polarised in the plane (E along y), B along y; the fields are what is asked for
        dict(name="pulse_2d_in_plane", kind="pulse", nx=1024, ny=512, pol="y", axion_bc="pml", precision="fp32", m=0.0,
             window=0, steps=100, every=0),
        # 3D laser pulse, absorbing along x, periodic across
        dict(name="laser_3d", kind="laser3d", nx=160, ny=96, nz=96, precision="fp64", m=0.0, steps=20, every=20),
        # the 3D box: an axion wave in uniform B makes photons, periodic
        dict(name="axion_3d", kind="axion3d", n=512, m=0.0, steps=100, every=100),
        # weak laser in a magnetised plasma, 4 macroparticles per cell
        dict(name="plasma_2d", kind="plasma", nx=12000, ny=100, ppc=4, spread=0.0, steps=8),
        # 2D requests of the serving stream advanced together, admitted, run, handed back
        dict(name="serve_2d", kind="serve", count=16, biggest=2048, steps=40),
    ]


def draw(rng):
    def span(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["line", "scan", "pulse", "pulse", "pulse", "axion2d", "laser3d", "axion3d", "plasma", "serve"])
    m = rng.choice([0.0, round(rng.uniform(1e-3, 1.0), 4)])
    if kind == "line":
        bc, prec = rng.choice([("periodic", "fp64"), ("periodic", "fp32"), ("pml", "fp64"), ("pml", "fp32")])
        return dict(kind=kind, nx=span(256, 16384), bc=bc, precision=prec, m=m, steps=span(100, 2000), every=rng.choice([0, 100, 500]))
    if kind == "scan":
        return dict(kind=kind, count=span(8, 512), steps=span(64, 512))
    if kind == "pulse":
        pol, abc, prec = rng.choice([("z", "pml", "fp64"), ("z", "pml", "fp32"), ("z", "outflow", "fp64"), ("y", "pml", "fp64"),
                                     ("y", "pml", "fp32")])
        most = 4096 if (pol, abc) == ("z", "pml") else 1024
        window = rng.choice([0, 16, 64]) if (pol, abc, prec) == ("z", "pml", "fp32") else 0
        nx, steps = span(256, most), span(20, 100)
        return dict(kind=kind, nx=nx, ny=span(128, most // 2), pol=pol, axion_bc=abc, precision=prec, m=m, window=window,
                    steps=steps, every=rng.choice([0, steps]) if pol == "z" else 0)
    if kind == "axion2d":
        return dict(kind=kind, nx=span(128, 1024), ny=span(128, 1024), axion_bc=rng.choice(["pml", "outflow"]), precision="fp64",
                    m=m, steps=span(20, 100), every=0)
    if kind == "laser3d":
        steps = span(5, 20)
        return dict(kind=kind, nx=span(64, 192), ny=span(32, 96), nz=span(32, 96), precision="fp64", m=m, steps=steps,
                    every=rng.choice([0, steps]))
    if kind == "axion3d":
        steps = span(10, 100)
        return dict(kind=kind, n=span(64, 400), m=m, steps=steps, every=rng.choice([0, steps]))
    if kind == "plasma":
        return dict(kind=kind, nx=span(400, 12000), ny=span(24, 100), ppc=rng.choice([1, 2, 4]), spread=rng.choice([0.0, 0.02]),
                    steps=span(4, 8))
    return dict(kind=kind, count=span(2, 16), biggest=span(512, 2048), steps=span(10, 40))


def _same(a):
    return (a, a)


def _setup(case, seed):
    """The numbers of one grid case: sizes, cell sizes, step, boundaries, waves (Sec. 3 set-ups)."""
    rng = np.random.default_rng([seed, 11])
    kind, dx = case["kind"], 1.0 / 32.0
    phase, amp = float(rng.uniform(0.0, K0)), float(rng.uniform(0.8, 1.2))
    s = dict(m=case["m"] * K0 if "m" in case else 0.0, g=1e-4, precision=case.get("precision", "fp64"), pml=20, smax=0.2,
             lo=(0.0, 0.0, 0.0), laser=None, axion=None, window=case.get("window", 0))
    per = _same("periodic")
    if kind == "line":
        nx = case["nx"]
        s.update(n=(nx, 1, 1), d=(dx, dx, dx), dt=0.95 * dx, B=(0.0, 1.0, 0.0), em=(_same(case["bc"]), per, per))
        s["ax"] = s["em"]
        L = nx * dx
        if case["bc"] == "periodic":
            k, c, dur = K0 * max(1, round(L)) / L, 0.0, 0.0
        else:
            k, c, dur = K0, L / 2.0, min(8.0, L / 8.0)
        s["laser"] = dict(amplitude=1e-3 * amp, k=(k, 0.0, 0.0), pol=(0.0, 1.0, 0.0), centre=(c, 0.0, 0.0), waist=0.0,
                          duration=dur, phase=phase)
    elif kind in ("pulse", "axion2d"):
        nx, ny = case["nx"], case["ny"]
        if kind == "axion2d":
            dx = 0.1
        Lx, Ly = nx * dx, ny * dx
        pml = _same("pml")
        s.update(n=(nx, ny, 1), d=(dx, dx, dx), dt=0.95 * dx / math.sqrt(2.0), lo=(0.0, -Ly / 2.0, 0.0), em=(pml, pml, per),
                 ax=(_same(case["axion_bc"]), _same(case["axion_bc"]), per))
        if kind == "axion2d":
            s.update(g=0.0, B=(0.0, 0.0, 0.0))
            s["axion"] = dict(amplitude=amp, k=(-K0, 0.0, 0.0), centre=(Lx / 2.0, 0.0, 0.0), waist=Ly / 8.0, length=Lx / 8.0,
                              speed=1.0, phase=phase)
        else:
            z = case["pol"] == "z"
            s["B"] = (0.0, 0.0, 1.0) if z else (0.0, 1.0, 0.0)
            s["laser"] = dict(amplitude=0.01 * amp, k=(K0, 0.0, 0.0), pol=(0.0, 0.0, 1.0) if z else (0.0, 1.0, 0.0),
                              centre=(min(16.0, Lx / 2.0), 0.0, 0.0), waist=min(4.0, Ly / 8.0), duration=min(8.0, Lx / 8.0),
                              phase=phase)
    elif kind == "laser3d":
        dx = 1.0 / 16.0
        n = (case["nx"], case["ny"], case["nz"])
        L = [c * dx for c in n]
        s.update(n=n, d=(dx, dx, dx), dt=0.95 * dx / math.sqrt(3.0), lo=(0.0, -L[1] / 2.0, -L[2] / 2.0), B=(0.0, 1.0, 0.0),
                 em=(_same("pml"), per, per), ax=(_same("pml"), per, per), pml=10)
        s["laser"] = dict(amplitude=0.01 * amp, k=(K0, 0.0, 0.0), pol=(0.0, 1.0, 0.0), centre=(L[0] / 2.0, 0.0, 0.0),
                          waist=min(L[1], L[2]) / 8.0, duration=L[0] / 8.0, phase=phase)
    elif kind == "axion3d":
        n, dx = case["n"], 1.0 / 16.0
        L = n * dx
        s.update(n=(n, n, n), d=(dx, dx, dx), dt=0.95 * dx / math.sqrt(3.0), B=(0.0, 1.0, 0.0), em=(per, per, per), ax=(per, per, per),
                 precision="fp32")
        s["axion"] = dict(amplitude=1e-2 * amp, k=(K0 * max(1, round(L)) / L, 0.0, 0.0), centre=(L / 2.0, L / 2.0, L / 2.0),
                          waist=L / 8.0, length=0.0, speed=1.0, phase=phase)
    elif kind == "plasma":
        nx, ny = case["nx"], case["ny"]
        d = (1.0 / 300.0, 1.0, 1.0)
        s.update(n=(nx, ny, 1), d=d, dt=0.95 / math.sqrt(1.0 / d[0] ** 2 + 1.0 / d[1] ** 2), lo=(-nx * d[0] / 2.0, -ny / 2.0, 0.0),
                 em=(per, per, per), ax=(per, per, per), m=0.0, g=0.0, density=3e-3 * K0 * K0)
        s["B"] = (0.0, 0.0, math.sqrt(s["density"]))
    return s


def _members(case, seed):
    """Uneven instances of one scan or serving case, drawn as the request stream draws them."""
    rng = np.random.default_rng([seed, 12])
    sizes = np.random.default_rng([case["count"], 13])  # the sizes belong to the case, the physics to the seed
    out = []
    for _ in range(case["count"]):
        q = dict(m=K0 * math.exp(rng.uniform(math.log(1e-3), math.log(2.0))), g=math.exp(rng.uniform(math.log(1e-6), math.log(1e-3))),
                 B0=math.exp(rng.uniform(math.log(0.1), math.log(10.0))))
        if case["kind"] == "scan":
            q["nx"] = int(round(math.exp(sizes.uniform(math.log(1024), math.log(65536)))))
        else:
            nx = int(round(math.exp(sizes.uniform(math.log(256), math.log(case["biggest"])))))
            q["nx"] = nx - nx % 2
            q["ny"] = q["nx"] // 2
        out.append(q)
    return out


def _beam(q):
    """A 2D conversion request: periodic along x, absorbing along y, a CW E_z beam, B along z."""
    dx = 1.0 / 32.0
    Lx, Ly = q["nx"] * dx, q["ny"] * dx
    per, pml = _same("periodic"), _same("pml")
    return dict(n=(q["nx"], q["ny"], 1), d=(dx, dx, dx), dt=0.95 * dx / math.sqrt(2.0), lo=(0.0, -Ly / 2.0, 0.0), m=q["m"], g=q["g"],
                B=(0.0, 0.0, q["B0"]), em=(per, pml, per), ax=(per, pml, per), pml=20, smax=0.2, precision="fp32", axion=None, window=0,
                laser=dict(amplitude=1e-3, k=(K0 * max(1, round(Lx)) / Lx, 0.0, 0.0), pol=(0.0, 0.0, 1.0), centre=(0.0, 0.0, 0.0),
                           waist=Ly / 8.0, duration=0.0, phase=0.0))


def _particles(case, s, seed):
    """Weights, positions, momenta of both orders (13 rows) and the pulse of the first-order fields."""
    n, d, lo, ppc = s["n"], s["d"], s["lo"], case["ppc"]
    gen = torch.Generator().manual_seed(seed + 14)
    cells = n[0] * n[1]
    count = cells * ppc
    rows = torch.zeros(13, count, dtype=torch.float64)
    rows[0] = s["density"] * d[0] * d[1] * d[2] / ppc
    cell = torch.arange(cells, dtype=torch.float64).repeat_interleave(ppc)
    j = torch.floor(cell / n[0])
    rows[1] = lo[0] + (cell - j * n[0] + torch.rand(count, generator=gen, dtype=torch.float64)) * d[0]
    rows[2] = lo[1] + (j + torch.rand(count, generator=gen, dtype=torch.float64)) * d[1]
    rows[3] = lo[2] + 0.5 * d[2]
    if case["spread"]:
        rows[4:7] = torch.randn(3, count, generator=gen, dtype=torch.float64) * case["spread"]
    rng = np.random.default_rng([seed, 15])
    A, xc = 1e-20 * s["B"][2], float(rng.uniform(-0.2, 0.0)) * n[0] * d[0]
    xe = lo[0] + (np.arange(n[0]) + 0.5) * d[0]
    y = lo[1] + (np.arange(n[1]) + 1.0) * d[1]
    pulse = lambda x: A * np.exp(-((x - xc) / 3.0) ** 2) * np.cos(K0 * (x - xc))  # noqa: E731
    trans = np.exp(-((y / (0.2 * n[1])) ** 2))[:, None]
    return rows, (trans * pulse(xe)[None])[None], (trans * pulse(xe + 0.5 * d[0])[None])[None]


# ---- through the solver ----

def _grid(s, every=0, capacity=0):
    spec = GridSpec(n=s["n"], d=s["d"], dt=s["dt"], lo=s["lo"], m=s["m"], g=s["g"], B_ext=s["B"], axion_bc=s["ax"], em_bc=s["em"],
                    pml_cells=s["pml"], pml_sigma_max_dt=s["smax"], precision=s["precision"])
    g = axp.Grid(spec, diag_every=every, diag_capacity=capacity)
    if s["laser"]:
        g.inject_laser(LaserSpec(**s["laser"]))
    if s["axion"]:
        g.inject_axion(AxionSpec(**s["axion"]))
    if s["window"]:
        g.set_moving_window(0, 1.0, s["window"], 0)
    return g


def _rows(g):
    """A device buffer for the whole state of an FP32 grid, and how many rows it holds."""
    n = [c for c in g.spec.n if c > 1][-1]
    return torch.empty(axp.axp_rows_bytes(g.h, n), dtype=torch.uint8, device="cuda"), n


def _parts(a, laser=True):
    """The 14 arrays of a state (14, cells), grouped by order."""
    out = {"order0": a[0:6]} if laser else {}
    out.update(order1=a[6:12], phi=a[12], second=a[13])
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "scan":
        members = _members(case, seed)
        b = batch.Batch(len(members), sum(q["nx"] for q in members), graphs=True)
        dx = 1.0 / 32.0
        slots = []
        for q in members:
            k = K0 * max(1, round(q["nx"] * dx)) / (q["nx"] * dx)
            slots.append(b.add(batch.instance_of(q["nx"], dx, 0.95 * dx, q["m"], q["g"], q["B0"], 0.0, 1e-3, k, 10**9)))
        b.set_tiling(64, 1664, 256)
        return dict(case=case, batch=b, slots=slots)
    if kind == "serve":
        grids = [_grid(_beam(q)) for q in _members(case, seed)]
        tiles = sum(group.tiles_of(g.spec.n[0], g.spec.n[1]) for g in grids)
        return dict(case=case, group=group.Group(len(grids), tiles, graphs=True), grids=grids, bufs=[_rows(g) for g in grids])
    s = _setup(case, seed)
    every = case.get("every", 0)
    g = _grid(s, every, case["steps"] // every + 1 if every else 0)
    st = dict(case=case, grid=g, every=every, laser=s["laser"] is not None or kind == "plasma")
    if kind == "plasma":
        rows, e1y, b1z = _particles(case, s, seed)
        g.write("E1y", e1y)
        g.write("B1z", b1z)
        r = rows.numpy()
        g.attach_particles(-1.0, 1.0, r[0], r[1:4], r[4:7], r[7:10], r[10:13])
        st["rows"] = torch.empty(13, rows.shape[1], dtype=torch.float64, pin_memory=True)
    if s["precision"] == "fp64":
        st["host"] = torch.empty(14, g.cells, dtype=torch.float64, pin_memory=True)
    else:
        st["buf"] = _rows(g)
    return st


def _pack(g, buf):
    axp.axp_pack_rows(g.h, 0, buf[1], buf[0].data_ptr(), buf[0].numel())
    return buf[0].view(torch.float32).view(14, g.cells)


def _pointer(t):
    return ctypes.cast(t.data_ptr(), ctypes.POINTER(ctypes.c_double))


def run(state):
    case = state["case"]
    if case["kind"] == "scan":
        b = state["batch"]
        b.run(case["steps"])
        rec = [[r["H_phi"], r["H_g0"], r["H_g1"]] for r in b.results(state["slots"])]
        phi = np.concatenate([b.read_state(slot, 6) for slot in state["slots"]])
        return dict(energies=np.array(rec, dtype=np.float32), phi=phi.astype(np.float32))
    if case["kind"] == "serve":
        grp = state["group"]
        members = [grp.add(g, case["steps"]) for g in state["grids"]]
        grp.run(case["steps"])
        for i in members:
            grp.remove(i)
        out = []
        for g, buf in zip(state["grids"], state["bufs"]):
            p = _parts(_pack(g, buf))
            out.append([p["order0"], p["order1"], p["phi"]])
        return out
    g = state["grid"]
    g.step(case["steps"])
    out = {}
    if state["every"]:
        rec = [[r["H_phi"], r["H_g0"], r["H_g1"]] for r in g.read_diagnostics()]
        out["energies"] = np.array(rec, dtype=np.float32 if "buf" in state else np.float64)
    if "buf" in state:
        out.update(_parts(_pack(g, state["buf"]), state["laser"]))
        return out
    host = state["host"]
    L = axp.lib()
    for f in range(14):
        if L.axp_read_field(g.h, f, _pointer(host[f]), 8 * g.cells) != axp.AXP_OK:
            raise RuntimeError("axp_read_field")
    out.update(_parts(host, state["laser"]))
    if "rows" in state:
        r = state["rows"]
        if L.axp_read_particles(g.h, _pointer(r), 8 * r.numel()) != axp.AXP_OK:
            raise RuntimeError("axp_read_particles")
        out.update(x0=r[1:4], u0=r[4:7], x1=r[7:10], u1=r[10:13])
    return out


def work(case):
    """Bytes: the state read once and written once.  Flops per cell and step: counted from the scheme
    for the components the set-up can excite (110 with a TM laser in 2D); about 700 per particle."""
    kind, steps = case["kind"], case["steps"]
    if kind in ("scan", "serve"):
        cells = sum(q["nx"] * q.get("ny", 1) for q in _members(case, 0))
        arrays, size, flops, parts = (8, 4, 60, 0) if kind == "scan" else (11, 4, 110, 0)
    else:
        s = _setup(case, 0)
        cells = s["n"][0] * s["n"][1] * s["n"][2]
        size = 4 if s["precision"] == "fp32" else 8
        arrays, flops = {"line": (8, 60), "pulse": (11, 110), "axion2d": (2, 10), "laser3d": (14, 200), "axion3d": (8, 90),
                         "plasma": (12, 100)}[kind]
        parts = cells * case["ppc"] if kind == "plasma" else 0
    return {"bytes": 2.0 * cells * arrays * size + 200.0 * parts, "flops": float(steps) * (cells * flops + parts * 700)}


# ---- the same in 64 bits, on whole arrays ----

class _Box:
    """One grid's arrays (nz, ny, nx), their neighbours under its boundaries, and its constants."""

    def __init__(self, s):
        self.s, self.n, self.d, self.dt, self.B = s, s["n"], s["d"], s["dt"], s["B"]
        self.m2, self.g = s["m"] ** 2, s["g"]
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.per = [s["em"][a][0] == "periodic" for a in range(3)]
        self.active = [c > 1 for c in self.n]
        self.sig_em, self.sig_ax = self._sigma(s["em"]), self._sigma(s["ax"])
        self.out = [(a, e) for a in range(3) for e in range(2) if s["ax"][a][e] == "outflow"]
        h = self.dt / 2.0
        self.ea, self.eb = (1.0 - self.sig_em * h / 2.0) / (1.0 + self.sig_em * h / 2.0), h / (1.0 + self.sig_em * h / 2.0)

    def _sigma(self, bc):
        N, top = self.s["pml"], 0.0
        for a in range(3):
            t = torch.zeros(self.n[a], dtype=torch.float64, device=self.dev)
            for e in range(2):
                if bc[a][e] == "pml" and N > 0:
                    c = torch.arange(self.n[a], device=self.dev)
                    c = c if e == 0 else self.n[a] - 1 - c
                    r = (1.0 - c.double() / N).clamp(min=0.0)
                    t = torch.maximum(t, r**3 * (self.s["smax"] / self.dt))
            if bool((t != 0).any()):
                t = t.view([-1 if 2 - a == q else 1 for q in range(3)])
                top = t if not torch.is_tensor(top) else torch.maximum(top, t)
        return top

    def zeros(self):
        return torch.zeros(self.n[2], self.n[1], self.n[0], dtype=torch.float64, device=self.dev)

    def edge(self, a, e):
        i = [slice(None)] * 3
        i[2 - a] = slice(0, 1) if e == 0 else slice(self.n[a] - 1, None)
        return tuple(i)

    def sh(self, F, a, step):
        """F one cell up (+1) or down (-1) along axis a; 0 beyond an edge that does not wrap."""
        if not torch.is_tensor(F) or not self.active[a]:
            return F
        R = torch.roll(F, -step, 2 - a)
        if not self.per[a]:
            R[self.edge(a, 1 if step > 0 else 0)] = 0.0
        return R

    def shp(self, F, ghost, a, step):
        """The same for the axion, whose outflow faces have a ghost plane."""
        R = self.sh(F, a, step)
        e = 1 if step > 0 else 0
        if (a, e) in self.out:
            R[self.edge(a, e)] = ghost[(a, e)]
        return R

    def pos(self, a, stag):
        x = self.s["lo"][a] + (torch.arange(self.n[a], dtype=torch.float64, device=self.dev) + (1.0 if stag else 0.5)) * self.d[a]
        return x.view([-1 if 2 - a == q else 1 for q in range(3)])

    def total(self, F):
        """Sum over the cells outside absorbing layers."""
        if not torch.is_tensor(F):
            return 0.0
        i = [slice(None)] * 3
        for a in range(3):
            N = self.s["pml"]
            lo, hi = ["pml" in (self.s["em"][a][e], self.s["ax"][a][e]) for e in range(2)]
            i[2 - a] = slice(N if lo else 0, self.n[a] - N if hi else self.n[a])
        return float(F.expand(self.n[2], self.n[1], self.n[0])[tuple(i)].sum())


class _Ragged(_Box):
    """Many periodic 1D boxes end to end, each with constants of its own."""

    def __init__(self, members):
        dx = 1.0 / 32.0
        per = _same("periodic")
        N = sum(q["nx"] for q in members)
        super().__init__(dict(n=(N, 1, 1), d=(dx, dx, dx), dt=0.95 * dx, m=0.0, g=0.0, B=(0.0, 0.0, 0.0), em=(per,) * 3, ax=(per,) * 3,
                              pml=0, smax=0.0, lo=(0.0, 0.0, 0.0)))
        size = torch.tensor([q["nx"] for q in members], device=self.dev)
        self.of = torch.repeat_interleave(torch.arange(len(members), device=self.dev), size)
        start = torch.cumsum(size, 0) - size
        self.at = torch.arange(N, device=self.dev) - start[self.of]
        self.first, self.last = start, start + size - 1
        flat = lambda v: torch.tensor(v, dtype=torch.float64, device=self.dev)[self.of].view(1, 1, -1)  # noqa: E731
        self.m2, self.g = flat([q["m"] ** 2 for q in members]), flat([q["g"] for q in members])
        self.B = (0.0, flat([q["B0"] for q in members]), 0.0)
        self.k = flat([K0 * max(1, round(q["nx"] * dx)) / (q["nx"] * dx) for q in members])
        self.count = len(members)

    def sh(self, F, a, step):
        if not torch.is_tensor(F) or a > 0:
            return F
        R = torch.roll(F, -step, 2)
        if step > 0:
            R[..., self.last] = F[..., self.first]
        else:
            R[..., self.first] = F[..., self.last]
        return R

    def total(self, F):
        if not torch.is_tensor(F):
            return np.zeros(self.count)
        out = torch.zeros(self.count, dtype=torch.float64, device=self.dev)
        return out.index_add_(0, self.of, F.view(-1)).cpu().numpy()


def _curl(b, F, step):
    """Forward (+1, of E) or backward (-1, of B) differences."""
    def diff(f, a):
        if not torch.is_tensor(f) or not b.active[a]:
            return 0.0
        return (b.sh(f, a, 1) - f) / b.d[a] if step > 0 else (f - b.sh(f, a, -1)) / b.d[a]

    return [diff(F[2], 1) - diff(F[1], 2), diff(F[0], 2) - diff(F[2], 0), diff(F[1], 0) - diff(F[0], 1)]


def _half(b, F, X):
    return [f if not torch.is_tensor(f) and not torch.is_tensor(x) else b.ea * f + b.eb * x for f, x in zip(F, X)]


def _ebar(b, E):
    return [0.5 * (E[a] + b.sh(E[a], a, -1)) for a in range(3)]


def _bbar(b, B):
    out = []
    for a in range(3):
        f, p, q = B[a], (a + 1) % 3, (a + 2) % 3
        out.append(0.25 * (f + b.sh(f, q, -1) + b.sh(f, p, -1) + b.sh(b.sh(f, p, -1), q, -1)) + b.B[a])
    return out


def _current(b, S):
    hi, lo = S["phi"], S["old"]
    mid, Dt = 0.5 * (hi + lo), (hi - lo) / b.dt
    gm = {f: 0.5 * (S["gc"][f] + S["go"][f]) for f in b.out}
    grad = [(b.shp(mid, gm, a, 1) - b.shp(mid, gm, a, -1)) / (2.0 * b.d[a]) if b.active[a] else 0.0 for a in range(3)]
    e, bb = _ebar(b, S["E0"]), _bbar(b, S["B0"])
    J = []
    for a in range(3):
        p, q = (a + 1) % 3, (a + 2) % 3
        P = Dt * bb[a] - (e[p] * grad[q] - e[q] * grad[p])
        up = b.sh(P, a, 1)
        if (a, 1) in b.out:  # beyond an outflow face only D_t phi B_ext is left
            up[b.edge(a, 1)] = (S["gc"][(a, 1)] - S["go"][(a, 1)]) / b.dt * b.B[a]
        J.append(0.5 * (P + up))
    return J


def _ehalf(b, S, J, orders):
    if 0 in orders:
        X = [x - j for x, j in zip(_curl(b, S["B0"], -1), S.get("j0", (0.0,) * 3))]
        S["E0"] = _half(b, S["E0"], X)
    if 1 in orders:
        X = [x - b.g * j - k for x, j, k in zip(_curl(b, S["B1"], -1), J, S.get("j1", (0.0,) * 3))]
        S["E1"] = _half(b, S["E1"], X)


def _bhalf(b, S):
    for o in "01":
        S["B" + o] = _half(b, S["B" + o], [-x for x in _curl(b, S["E" + o], 1)])


def _axion(b, S):
    e, bb = _ebar(b, S["E0"]), _bbar(b, S["B0"])
    src = b.g * sum(x * y for x, y in zip(e, bb))
    ph, old, dt = S["phi"], S["old"], b.dt
    lap = 0.0
    for a in range(3):
        if b.active[a]:
            lap = lap + (b.shp(ph, S["gc"], a, 1) + b.shp(ph, S["gc"], a, -1) - 2.0 * ph) / b.d[a] ** 2
    sig = b.sig_ax
    Y = src - b.m2 * ph + lap - sig * sig * ph
    new = (dt * dt * Y + sig * dt * old + 2.0 * ph - old) / (1.0 + sig * dt)
    ghost = {}
    for a, side in b.out:  # the one-way and the wave equation at the ghost
        r = dt / b.d[a]
        gc, go, p0 = S["gc"][(a, side)], S["go"][(a, side)], ph[b.edge(a, side)]
        Sg = 0.0
        if side == 1 and torch.is_tensor(S["E0"][a]):
            Sg = b.g * 0.5 * S["E0"][a][b.edge(a, 1)] * b.B[a]
        V = (-2.0 * gc + 2.0 * go - dt * dt * (Sg - b.m2 * gc) + r * p0 - r * r * (p0 - 2.0 * gc)) / (r + r * r)
        ghost[(a, side)] = go + r * (p0 - V)
    S.update(phi=new, old=ph, gc=ghost, go=S["gc"])


def _energies(b, S):
    mid, Dt = 0.5 * (S["phi"] + S["old"]), (S["phi"] - S["old"]) / b.dt
    gm = {f: 0.5 * (S["gc"][f] + S["go"][f]) for f in b.out}
    u = Dt * Dt + b.m2 * mid * mid
    for a in range(3):
        if b.active[a]:
            u = u + ((b.shp(mid, gm, a, 1) - mid) / b.d[a]) ** 2
    w = 0.5 * b.d[0] * b.d[1] * b.d[2]
    sq = lambda F: sum(f * f for f in F)  # noqa: E731
    return [b.total(u) * w, b.total(sq(S["E0"]) + sq(S["B0"])) * w, b.total(sq(S["E1"]) + sq(S["B1"])) * w]


def _start(b, s):
    """Fields at t = 0: the laser as the scheme's own eigenmode, the axion at t = +dt/2 and -dt/2."""
    S = dict(E0=[0.0] * 3, B0=[0.0] * 3, E1=[0.0] * 3, B1=[0.0] * 3, phi=b.zeros(), old=b.zeros(), gc={}, go={})

    def wave(w, stag):
        x = [b.pos(a, stag == a) - w["centre"][a] for a in range(3)]
        k = math.sqrt(sum(c * c for c in w["k"]))
        xi = sum(w["k"][a] / k * x[a] for a in range(3))
        r2 = x[0] ** 2 + x[1] ** 2 + x[2] ** 2 - xi * xi
        across = torch.exp(-r2 / w["waist"] ** 2) if w["waist"] > 0 else 1.0
        return xi, across, sum(w["k"][a] * x[a] for a in range(3)) + w["phase"]

    def big_k(w):
        return math.sqrt(sum((2.0 / b.d[a] * math.sin(w["k"][a] * b.d[a] / 2.0)) ** 2 for a in range(3)))

    if s["laser"]:
        w = s["laser"]
        K = big_k(w)
        length = w["duration"] / math.sqrt(2.0 * math.log(2.0))
        F = [0.0] * 3
        for a in range(3):
            if w["pol"][a]:
                xi, across, ph = wave(w, a)
                env = w["amplitude"] * w["pol"][a] * across * (torch.exp(-((xi / length) ** 2)) if length > 0 else 1.0)
                S["E0"][a] = b.zeros() + env * torch.cos(ph)
                F[a] = b.zeros() + env * torch.sin(ph) / (math.sqrt(1.0 - (b.dt * K / 2.0) ** 2) * K)
        S["B0"] = _curl(b, F, 1)
    if s["axion"]:
        w = s["axion"]
        om = math.acos(1.0 - b.dt**2 * (big_k(w) ** 2 + b.m2) / 2.0) / b.dt
        xi, across, ph = wave(w, None)

        def at(t, xi, across, ph):
            along = torch.exp(-(((xi - w["speed"] * t) / w["length"]) ** 2)) if w["length"] > 0 else 1.0
            return w["amplitude"] * across * along * torch.sin(ph - om * t)

        S["phi"], S["old"] = b.zeros() + at(0.5 * b.dt, xi, across, ph), b.zeros() + at(-0.5 * b.dt, xi, across, ph)
    for a, e in b.out:
        for name, t in (("gc", 0.5), ("go", -0.5)):
            if s["axion"]:
                keep = b.pos
                b.pos = lambda q, st, a=a, e=e: (keep(q, st)[b.edge(a, e)] + (b.d[a] if e else -b.d[a])) if q == a else keep(q, st)
                S[name][(a, e)] = at(t * b.dt, *wave(s["axion"], None)) + 0.0 * S["phi"][b.edge(a, e)]
                b.pos = keep
            else:
                S[name][(a, e)] = 0.0 * S["phi"][b.edge(a, e)]
    return S


def _advance(b, S, steps, every=0, window=0, push=None):
    energies, travel = [], S.get("travel", 0.0)
    J = _current(b, S)
    for k in range(steps):
        _ehalf(b, S, J, (0, 1))
        _bhalf(b, S)
        _axion(b, S)
        if push is not None:
            push()
        _bhalf(b, S)
        _ehalf(b, S, None, (0,))
        J = _current(b, S)
        _ehalf(b, S, J, (1,))
        if every and (k + 1) % every == 0:
            energies.append(_energies(b, S))
        if window:
            travel += b.dt / b.d[0]
            if travel >= window - 1e-9:
                travel -= window
                move = lambda f: torch.cat([f[..., window:], torch.zeros_like(f[..., :window])], -1) if torch.is_tensor(f) else f  # noqa: E731
                for name in ("E0", "B0", "E1", "B1"):
                    S[name] = [move(f) for f in S[name]]
                S["phi"], S["old"] = move(S["phi"]), move(S["old"])
                J = _current(b, S)
    return J, energies


def _state(b, S, J, staggered):
    """The 14 arrays; E half a step ahead and the axion's increment where the FP32 kernels hold them so."""
    if staggered:
        _ehalf(b, S, J, (0, 1))
    n = b.n[0] * b.n[1] * b.n[2]
    out = torch.zeros(14, n, dtype=torch.float64, device=b.dev)
    for i, f in enumerate(S["E0"] + S["B0"] + S["E1"] + S["B1"] + [S["phi"], S["phi"] - S["old"] if staggered else S["old"]]):
        if torch.is_tensor(f):
            out[i] = f.expand(b.n[2], b.n[1], b.n[0]).reshape(-1)
    return out


class _Plasma:
    """Macroparticles of Sec. 2.2: quadratic spline, Boris push of order 0 and its first-order part."""

    def __init__(self, b, rows, q=-1.0, m=1.0):
        self.b, self.q, self.m = b, q, m
        r = rows.to(b.dev)
        self.w, self.x0, self.u0, self.x1, self.u1 = r[0], list(r[1:4]), list(r[4:7]), list(r[7:10]), list(r[10:13])

    def nodes(self, x0, x1, kind, a):
        """(flat index, weight S, weight dS . x1) of the nodes of component a of E (kind 1) or B (2)."""
        b, ax = self.b, []
        for c in (0, 1):
            face = (c == a) == (kind == 1)
            xi = (x0[c] - b.s["lo"][c]) / b.d[c] - (1.0 if face else 0.5)
            near = torch.floor(xi + 0.5)
            e = xi - near
            W = (0.5 * (0.5 - e) ** 2, 0.75 - e * e, 0.5 * (0.5 + e) ** 2)
            D = (-(0.5 - e) / b.d[c], -2.0 * e / b.d[c], (0.5 + e) / b.d[c])
            ax.append([((near.long() + t - 1) % b.n[c], W[t], D[t] * x1[c]) for t in range(3)])
        for jy, wy, dy in ax[1]:
            for ix, wx, dx in ax[0]:
                yield ix + b.n[0] * jy, wx * wy, dx * wy + wx * dy

    def gather(self, F0, F1, kind, a, ext):
        f0, fp = ext, 0.0
        for at, s, ds in self.nodes(self.x0, self.x1, kind, a):
            for F, w, first in ((F0[a], s, False), (F0[a], ds, True), (F1[a], s, True)):
                if torch.is_tensor(F):
                    v = w * F.reshape(-1)[at]
                    f0, fp = (f0, fp + v) if first else (f0 + v, fp)
        return f0 + torch.zeros_like(self.w), fp + torch.zeros_like(self.w)

    def velocity(self):
        g2 = 1.0 + sum(u * u for u in self.u0)
        g = torch.sqrt(g2)
        uu = sum(u * v for u, v in zip(self.u0, self.u1))
        return [u / g for u in self.u0], [(g2 * v - u * uu) / (g * g2) for u, v in zip(self.u0, self.u1)]

    def deposit(self, S, x0, x1, v0, v1):
        b = self.b
        k = self.q * self.w / (b.d[0] * b.d[1] * b.d[2])
        S["j0"], S["j1"] = [b.zeros() for _ in range(3)], [b.zeros() for _ in range(3)]
        for a in range(3):
            for at, s, ds in self.nodes(x0, x1, 1, a):
                S["j0"][a].view(-1).index_add_(0, at, k * s * v0[a])
                S["j1"][a].view(-1).index_add_(0, at, k * (ds * v0[a] + s * v1[a]))

    def drift(self, t, v0, v1):
        b = self.b
        for a in range(3):
            x = self.x0[a] + t * v0[a]
            if b.active[a]:
                L, lo = b.n[a] * b.d[a], b.s["lo"][a]
                x = torch.where(x >= lo + L, x - L, torch.where(x < lo, x + L, x))
            self.x0[a], self.x1[a] = x, self.x1[a] + t * v1[a]

    def begin(self, S):
        v0, v1 = self.velocity()
        self.deposit(S, self.x0, self.x1, v0, v1)
        self.drift(self.b.dt / 2.0, v0, v1)

    def push(self, S):
        b = self.b
        h = self.q / self.m * b.dt / 2.0
        cross = lambda p, q: [p[1] * q[2] - p[2] * q[1], p[2] * q[0] - p[0] * q[2], p[0] * q[1] - p[1] * q[0]]  # noqa: E731
        dot = lambda p, q: p[0] * q[0] + p[1] * q[1] + p[2] * q[2]  # noqa: E731
        add = lambda *v: [sum(c) for c in zip(*v)]  # noqa: E731
        E, Ep = zip(*[self.gather(S["E0"], S["E1"], 1, a, 0.0) for a in range(3)])
        B, Bp = zip(*[self.gather(S["B0"], S["B1"], 2, a, b.B[a]) for a in range(3)])
        um, dm = [u + h * e for u, e in zip(self.u0, E)], [u + h * e for u, e in zip(self.u1, Ep)]
        g = torch.sqrt(1.0 + dot(um, um))
        dg = dot(um, dm) / g
        t = [h * x / g for x in B]
        dt = [h * x / g - y * dg / g for x, y in zip(Bp, t)]
        up, dup = add(um, cross(um, t)), add(dm, cross(dm, t), cross(um, dt))
        i = 1.0 + dot(t, t)
        s = [2.0 * x / i for x in t]
        ds = [2.0 * y / i - 2.0 * x * (2.0 * dot(t, dt)) / (i * i) for x, y in zip(t, dt)]
        self.u0 = add(um, cross(up, s), [h * e for e in E])
        self.u1 = add(dm, cross(dup, s), cross(up, ds), [h * e for e in Ep])
        v0, v1 = self.velocity()
        self.deposit(S, [x + 0.5 * b.dt * v for x, v in zip(self.x0, v0)], [x + 0.5 * b.dt * v for x, v in zip(self.x1, v1)], v0, v1)
        self.drift(b.dt, v0, v1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "scan":
        b = _Ragged(_members(case, seed))
        x = (b.at.view(1, 1, -1) + 0.5) * b.d[0]
        K = 2.0 / b.d[0] * torch.sin(b.k * b.d[0] / 2.0)
        S = dict(E0=[0.0, 1e-3 * torch.cos(b.k * x), 0.0], E1=[0.0] * 3, B1=[0.0] * 3, phi=b.zeros(), old=b.zeros(), gc={}, go={})
        S["B0"] = _curl(b, [0.0, 1e-3 * torch.sin(b.k * x) / (torch.sqrt(1.0 - (b.dt * K / 2.0) ** 2) * K), 0.0], 1)
        _advance(b, S, case["steps"])
        return dict(energies=np.stack(_energies(b, S), 1), phi=S["phi"].view(-1))
    if kind == "serve":
        out = []
        for q in _members(case, seed):
            s = _beam(q)
            b = _Box(s)
            S = _start(b, s)
            J, _ = _advance(b, S, case["steps"])
            p = _parts(_state(b, S, J, True))
            out.append([p["order0"], p["order1"], p["phi"]])
        return out
    s = _setup(case, seed)
    b = _Box(s)
    S = _start(b, s)
    push = P = None
    if kind == "plasma":
        rows, e1y, b1z = _particles(case, s, seed)
        S["E1"][1], S["B1"][2] = torch.from_numpy(e1y).to(b.dev), torch.from_numpy(b1z).to(b.dev)
        P = _Plasma(b, rows)
        P.begin(S)
        push = lambda: P.push(S)  # noqa: E731
    J, energies = _advance(b, S, case["steps"], case.get("every", 0), s["window"], push)
    out = {"energies": np.array(energies)} if energies else {}
    out.update(_parts(_state(b, S, J, s["precision"] == "fp32"), s["laser"] is not None or kind == "plasma"))
    if P is not None:
        P.drift(-b.dt / 2.0, *P.velocity())
        out.update(x0=torch.stack(P.x0), u0=torch.stack(P.u0), x1=torch.stack(P.x1), u1=torch.stack(P.u1))
    return out
