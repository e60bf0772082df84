"""Performance cases of the coupled LB/FD step, through the public binding
(``paper_2304_05657_gb300.lbfd``, ``.channels``).

A case is one call pattern of a user's program: the handle (grid, geometry,
mechanism, state on the device) is what such a program keeps, a pass advances
it and reads the result back into a host buffer the program owns.

- listed():            the named cases, with what each stands for
- draw(rng):           one more case of the same ranges
- prepare(case, seed): geometry from the case, fields from the seed, a handle
- run(state):          one pass
- work(case):          bytes and operations a pass cannot do without
- exact(case, seed):   the same outputs by a restatement of the step in plain
                       torch FP64 (definitional forms, no library code)

Sizes are those of the benchmark's workloads, the tests and their profiling
sizes, or odd ones between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2304_05657_gb300 import channels, inputs, lbfd

DEV = "cuda"
CS2 = 1.0 / 3.0
NSP = 5


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the plain FP64 verification channel, single-step launches, the
        # library's default kernel: what a first user runs
        dict(name="channel fp64", kind="channel", nx=256, ny=32, walls="adiabatic", precision="fp64", launch="step",
             tuned=False, steps=100),
        # the same channel in production arithmetic: latency and launches are all
        dict(name="channel mixed graph", kind="channel", nx=256, ny=32, walls="adiabatic", precision="mixed",
             launch="graph", tuned=True, steps=200),
        # inflow control holding a flame in a small channel: short bursts of
        # steps between reductions and a changed inlet velocity
        dict(name="held flame fp64", kind="hold", nx=120, ny=12, walls="adiabatic", precision="fp64", launch="step",
             tuned=False, steps=200, every=50),
        # the channel study: 16 channels of uneven width in one domain, the
        # autotuned kernel, graph launches (the 2-D benchmark workload)
        dict(name="channel study mixed", kind="batch", widths=",".join(str(16 + 12 * j) for j in range(16)),
             length=1024, precision="mixed", launch="graph", tuned=True, steps=50),
        # a small FP64 study with odd widths and length and its per-channel
        # observables (flame position, reaction front per column)
        dict(name="odd study fp64", kind="batch", widths="17,33,65", length=301, precision="fp64", launch="graph",
             tuned=True, steps=50),
        # the slotted burner: 2-D with curved rows of solids in the flow
        dict(name="burner mixed", kind="burner", nx=2048, ny=512, precision="mixed", launch="graph", tuned=True,
             steps=50),
        # 3-D porous burner, production arithmetic: profiling size and largest
        dict(name="packing mixed small", kind="packing", nx=128, ny=64, nz=64, precision="mixed", launch="graph",
             tuned=True, steps=20),
        dict(name="packing mixed large", kind="packing", nx=256, ny=128, nz=128, precision="mixed", launch="step",
             tuned=True, steps=25),
        # 3-D in FP64 with odd extents, default kernel, plus the flame position
        dict(name="odd packing fp64", kind="packing", nx=101, ny=53, nz=47, precision="fp64", launch="step",
             tuned=False, steps=5),
        # gradients of the flame position: discrete adjoint and forward mode
        dict(name="adjoint fp64", kind="adjoint", nx=512, ny=64, walls="isothermal", precision="fp64", launch="step",
             tuned=False, steps=100, every=25),
        dict(name="tangent fp64", kind="channel", nx=512, ny=64, walls="isothermal", precision="tangent",
             launch="step", tuned=False, steps=25),
        dict(name="tangent mixed", kind="channel", nx=512, ny=64, walls="isothermal", precision="tangent_mixed",
             launch="step", tuned=False, steps=50),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["channel", "channel", "hold", "batch", "batch", "burner", "packing", "packing", "adjoint",
                       "tangent"])
    prec = rng.choice(["mixed", "mixed", "fp64"])
    walls = rng.choice(["adiabatic", "isothermal"])
    tuned = rng.random() < 0.5
    launch = rng.choice(["step", "graph"])
    if kind == "channel":
        return dict(kind=kind, nx=_log(rng, 64, 1024), ny=_log(rng, 12, 200), walls=walls, precision=prec,
                    launch=rng.choice(["step", "graph", "persistent"]), tuned=tuned,
                    steps=_log(rng, 10, 200 if prec == "mixed" else 60))
    if kind == "hold":
        return dict(kind=kind, nx=_log(rng, 80, 400), ny=_log(rng, 9, 64), walls="adiabatic", precision="fp64",
                    launch="step", tuned=False, steps=100, every=_log(rng, 10, 50))
    if kind == "batch":
        widths = [_log(rng, 9, 196) for _ in range(rng.randint(2, 12))]
        return dict(kind=kind, widths=",".join(map(str, widths)), length=_log(rng, 100, 1024), precision=prec,
                    launch=rng.choice(["step", "graph", "persistent"]), tuned=tuned,
                    steps=_log(rng, 10, 50) if prec == "mixed" else _log(rng, 3, 12))
    if kind == "burner":
        return dict(kind=kind, nx=_log(rng, 256, 2048), ny=64 * _log(rng, 2, 8), precision=prec, launch=launch,
                    tuned=tuned, steps=_log(rng, 10, 50) if prec == "mixed" else _log(rng, 2, 5))
    if kind == "packing":
        ny, nz = _log(rng, 33, 96), _log(rng, 33, 96)
        return dict(kind=kind, nx=_log(rng, 80, 224), ny=ny, nz=nz, precision=prec, launch=launch, tuned=tuned,
                    steps=_log(rng, 5, 20) if prec == "mixed" else _log(rng, 1, 3))
    if kind == "adjoint":
        n = _log(rng, 10, 100)
        return dict(kind=kind, nx=_log(rng, 64, 512), ny=_log(rng, 16, 64), walls=walls, precision="fp64",
                    launch="step", tuned=False, steps=n, every=max(1, n // rng.randint(1, 4)))
    return dict(kind="channel", nx=_log(rng, 64, 512), ny=_log(rng, 16, 64), walls=walls,
                precision=rng.choice(["tangent", "tangent_mixed"]), launch="step", tuned=False,
                steps=_log(rng, 5, 25))


# ---------------------------------------------------------------------------
# geometry and fields
# ---------------------------------------------------------------------------

def _geometry(case):
    """(cfg, solid[nz, ny, nx] bool on the GPU, hot band (x0, x1, T_hot), rows
    of the channels or None)."""
    kind = case["kind"]
    rows = None
    if kind in ("channel", "hold", "adjoint"):
        wt = "wall_" + case["walls"]
        nx, ny, nz = case["nx"], case["ny"], 1
        cfg = inputs.base_config(dim=2, nx=nx, ny=ny, u_in=0.01,
                                 bc=["inlet", "outlet_pressure", wt, wt, "periodic", "periodic"])
        band = (nx // 3, nx // 3 + 20, 2000.0) if kind == "hold" else (0, 20, 2000.0)
        solid = torch.zeros((1, ny, nx), dtype=torch.bool, device=DEV)
    elif kind == "batch":
        widths = [int(w) for w in case["widths"].split(",")]
        nx, ny, nz = case["length"], sum(widths) + len(widths) - 1, 1
        cfg = inputs.base_config(dim=2, nx=nx, ny=ny, u_in=0.0,
                                 bc=["wall_adiabatic", "outlet_pressure", "wall_isothermal", "wall_isothermal",
                                     "periodic", "periodic"])
        solid = torch.zeros((1, ny, nx), dtype=torch.bool, device=DEV)
        rows, y = [], 0
        for w in widths:
            rows.append((y, y + w))
            if y + w < ny:
                solid[0, y + w] = True
            y += w + 1
        band = (0, 20, 2000.0)
    elif kind == "burner":
        nx, ny, nz = case["nx"], case["ny"], 1
        cfg = inputs.base_config(dim=2, nx=nx, ny=ny, u_in=0.02, T_solid=373.0, Y_in=inputs.premixed_Y(0.8),
                                 bc=["inlet", "outlet_pressure"] + ["periodic"] * 4)
        x0, x1 = nx // 4, nx // 4 + max(64, nx // 128 * 64)
        yy = torch.arange(ny, device=DEV, dtype=torch.float64)[:, None] + 0.5
        xx = torch.arange(nx, device=DEV, dtype=torch.float64)[None, :] + 0.5
        s = torch.zeros((ny, nx), dtype=torch.bool, device=DEV)
        for col, xc in enumerate(np.arange(x0 + 32.0, x1, 64.0)):
            dy = torch.remainder(yy - 32.0 * (col % 2) + 32.0, 64.0) - 32.0  # pitch 64, alternate rows offset
            s |= (xx - float(xc)) ** 2 + dy ** 2 <= 400.0
        solid = s[None]
        band = (x1, x1 + 20, 2000.0)
    else:  # packing of overlapping spheres, porosity about 0.80, periodic in y and z
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        cfg = inputs.base_config(dim=3, nx=nx, ny=ny, nz=nz, u_in=0.01,
                                 bc=["inlet", "outlet_pressure"] + ["periodic"] * 4)
        x0, x1 = nx // 8, nx - nx // 8
        rng = np.random.Generator(np.random.PCG64(20230411))
        r3 = (16.0 ** 4 - 8.0 ** 4) / 4.0 / 8.0  # mean cube of a radius uniform in [8, 16]
        n = int(round(-math.log(0.80) * (x1 - x0) * ny * nz / (4.0 / 3.0 * math.pi * r3)))
        solid = torch.zeros((nz, ny, nx), dtype=torch.bool, device=DEV)
        ax = [torch.arange(m, device=DEV, dtype=torch.float32) + 0.5 for m in (nz, ny, nx)]
        for _ in range(max(n, 1)):
            r = float(rng.uniform(8.0, 16.0))
            cx, cy, cz = rng.uniform(x0 + r, x1 - r), rng.uniform(0, ny), rng.uniform(0, nz)
            dz = torch.remainder(ax[0] - cz + nz / 2.0, float(nz)) - nz / 2.0
            dy = torch.remainder(ax[1] - cy + ny / 2.0, float(ny)) - ny / 2.0
            dx = ax[2] - cx
            solid |= dz[:, None, None] ** 2 + dy[None, :, None] ** 2 + dx[None, None, :] ** 2 <= r * r
        band = (x1, x1 + 20, cfg["T_in"] + cfg["Q"] * cfg["Y_in"][inputs.FUEL] / cfg["cp"])
    cfg["precision"] = case["precision"]
    return cfg, solid, band, rows


def _wall_taper(cfg, solid):
    """0 next to isothermal boundaries, 1 four cells away (the hot band and
    the fluctuations fade out there, as in the repository's own inputs)."""
    bc = cfg["bc"]
    near = solid.to(torch.float32)[None, None]
    out = torch.zeros_like(near)
    pad = [1, 1, 1, 1] + ([1, 1] if cfg["dim"] == 3 else [0, 0])
    m = near
    for _ in range(4):
        out += m
        q = torch.nn.functional.pad(m, pad, mode="constant", value=0.0)
        for a, dimn in ((0, 4), (1, 3), (2, 2)):
            if a >= cfg["dim"]:
                continue
            last = q.shape[dimn] - 1
            lo, hi = q.select(dimn, 0), q.select(dimn, last)
            if bc[2 * a] == "periodic":
                lo.copy_(q.select(dimn, last - 1))
                hi.copy_(q.select(dimn, 1))
            else:
                if bc[2 * a] == "wall_isothermal":
                    lo.fill_(1.0)
                if bc[2 * a + 1] == "wall_isothermal":
                    hi.fill_(1.0)
        k = (3 if cfg["dim"] == 3 else 1, 3, 3)
        m = torch.nn.functional.max_pool3d(q, k, stride=1)
    out += m
    return (1.0 - out[0, 0] / 5.0).clamp(0.0, 1.0).to(torch.float64)


def _directions(dim):
    n = 27 if dim == 3 else 9
    return [(i % 3 - 1, (i // 3) % 3 - 1, i // 9 - 1 if dim == 3 else 0) for i in range(n)]


def _weights(dim):
    w = {0: 2.0 / 3.0, 1: 1.0 / 6.0, -1: 1.0 / 6.0}
    return [w[c[0]] * w[c[1]] * (w[c[2]] if dim == 3 else 1.0) for c in _directions(dim)]


def _fields(cfg, solid, band, seed):
    """g[Q, N], T[N], Y[5, N] in FP64 on the GPU: unburnt mixture with a hot
    band of burnt gas, smooth fluctuations drawn from the seed, and the
    populations of a smooth low-Mach flow (equilibrium)."""
    dim, nx, ny, nz = cfg["dim"], cfg["nx"], cfg["ny"], cfg["nz"]
    gen = torch.Generator(device="cpu").manual_seed(int(seed) * 7919 + 17)
    f64 = dict(dtype=torch.float64, device=DEV)
    x = (torch.arange(nx, **f64) + 0.5)[None, None, :]
    y = (torch.arange(ny, **f64) + 0.5)[None, :, None]
    z = (torch.arange(nz, **f64) + 0.5)[:, None, None]

    def noise():
        s = torch.zeros((nz, ny, nx), **f64)
        for _ in range(5):
            k = [int(torch.randint(0, 4, (1,), generator=gen)) for _ in range(3)]
            ph = float(torch.rand(1, generator=gen)) * 2.0 * math.pi
            a = float(torch.rand(1, generator=gen)) - 0.5
            s += a * torch.cos(2.0 * math.pi * (k[0] * x / nx + k[1] * y / ny + (k[2] * z / nz if nz > 1 else 0.0)) + ph)
        return s

    taper = _wall_taper(cfg, solid)
    x0, x1, T_hot = band
    left = torch.ones_like(x) if x0 <= 0 else 0.5 * (1.0 + torch.tanh((x - x0) / 1.5))
    prof = left * 0.5 * (1.0 - torch.tanh((x - x1) / 1.5)) * taper
    prof = (prof * (1.0 + 0.05 * noise())).clamp(0.0, 1.0)
    fluid = (~solid).to(torch.float64)
    T = cfg["T_in"] + (T_hot - cfg["T_in"]) * prof + 8.0 * noise() * taper
    T = torch.where(solid, torch.full_like(T, cfg["T_solid"]), T)
    Yu = torch.tensor(cfg["Y_in"], **f64)[:, None, None, None]
    Yb = torch.tensor(inputs.burnt_Y(cfg["Y_in"]), **f64)[:, None, None, None]
    mix = (prof + 0.02 * (1.0 + noise()) * taper).clamp(0.0, 1.0)
    Y = Yu + (Yb - Yu) * mix
    W = torch.tensor(cfg["W"], **f64)[:, None, None, None]
    invW_in = sum(a / b for a, b in zip(cfg["Y_in"], cfg["W"]))
    rho = cfg["T_in"] * invW_in / (T * (Y / W).sum(0))
    U = max(cfg["u_in"], 0.01)
    u = [U * (1.0 + 0.3 * noise()), 0.3 * U * noise(), 0.3 * U * noise() if dim == 3 else torch.zeros_like(T)]
    P = 5e-4 * noise()
    uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
    g = []
    for c, w in zip(_directions(dim), _weights(dim)):
        cu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2]
        g.append((w * (P + rho * (cu + 1.5 * cu * cu - 0.5 * uu)) * fluid).reshape(-1))
    return torch.stack(g), T.reshape(-1), Y.reshape(NSP, -1)


STORE = {"fp64": torch.float64, "mixed": torch.float32, "tangent": torch.float64, "tangent_mixed": torch.float32}


def prepare(case, seed):
    cfg, solid, band, rows = _geometry(case)
    g, T, Y = _fields(cfg, solid, band, seed)
    stream = torch.cuda.current_stream()
    if case["kind"] == "batch":
        widths = [b - a for a, b in rows]
        s, rows = lbfd.batch_create(widths, case["length"], cfg, stream=stream)
    else:
        s = lbfd.Solver(cfg, solid.to(torch.uint8).cpu().numpy(), stream=stream)
    dt = STORE[case["precision"]]
    tan = case["precision"].startswith("tangent")
    if tan:
        s.set_state(T.cpu().numpy(), Y.cpu().numpy(), g.cpu().numpy())
    else:
        raw = torch.cat([g, T[None], Y]).to(dt).cpu().contiguous()
        s.set_state_raw(raw.data_ptr(), raw.numel() * raw.element_size())
    if case["tuned"]:
        s.autotune(5)
    shape = (s.Q + 1 + NSP, s.N) + ((5,) if tan else ())
    host = torch.empty(shape, dtype=dt, pin_memory=True)
    st = dict(case=case, s=s, rows=rows, host=host)
    if case["kind"] == "hold":
        st["control"] = channels.InflowController(x_target=s.diagnostics()["x_f"] + 5.0)
    if case["kind"] == "adjoint":
        s.adjoint_setup(case["every"])
    return st


def _state_out(st):
    """The whole state through the pinned host buffer: populations, T, Y."""
    s, host = st["s"], st["host"]
    s.get_state_raw(host.data_ptr(), host.numel() * host.element_size())
    Q = s.Q
    return {"g": host[:Q], "T": host[Q], "Y": host[Q + 1:]}


DIAG = ("x_f", "mass", "heat_release", "fuel_consumption", "T_max", "x_hrr_max", "n_nonfinite", "n_fluid")


def run(st):
    case, s = st["case"], st["s"]
    kind, n = case["kind"], case["steps"]
    out = {}
    if kind == "hold":
        hist = channels.hold_flame(s, st["control"], steps=n, every=case["every"])
        out["history"] = np.array([h[1:] for h in hist], dtype=np.float64)  # (x_f, u_in) per update
    elif kind == "adjoint":
        J, grad = s.adjoint_run(n)
        out["J"], out["grad"] = J, grad
    elif case["launch"] == "graph":
        s.step_graph(n)
    elif case["launch"] == "persistent":
        s.step_persistent(n)
    else:
        s.step(n)
    if case["precision"] == "tangent":
        out["J"], out["grad"] = s.gradient()
    if kind == "batch" and case["precision"] == "fp64":
        out["diag"] = np.array([[d[k] for k in DIAG] for d in channels.channel_diagnostics(s, st["rows"])])
        out["front"] = np.stack([np.stack(s.column_peaks(r)) for r in st["rows"]])
    if kind == "packing" and case["precision"] == "fp64":
        out["flame"] = np.array(s.flame_position())
    out["state"] = _state_out(st)
    return out


# ---------------------------------------------------------------------------
# work: the state read once and written once per step (it is the interface
# between steps of this explicit scheme) and once to the host per pass, and
# the floating-point operations of the scheme as written
# ---------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "packing":
        cells, dim = case["nx"] * case["ny"] * case["nz"] * 0.85, 3
    elif kind == "batch":
        cells, dim = case["length"] * sum(int(w) for w in case["widths"].split(",")), 2
    elif kind == "burner":
        cells, dim = case["nx"] * case["ny"] * 0.85, 2
    else:
        cells, dim = case["nx"] * case["ny"], 2
    planes = (27 if dim == 3 else 9) + 1 + NSP
    e = 4 if case["precision"] in ("mixed", "tangent_mixed") else 8
    tan = 5 if case["precision"].startswith("tangent") else 1
    n = case["steps"]
    # per axis: rho, 1/W and T lines (~55), and per species the mole-fraction
    # and mass-fraction lines, WENO3 and the fluxes (~66); collision ~300
    # (D2Q9) or ~1150 (D3Q27); Arrhenius and the update ~40
    flops = dim * (55 + 66 * NSP) + (300 if dim == 2 else 1150) + 40
    state = planes * e * tan * cells
    b = n * (2 * state + cells) + state
    f = n * flops * cells * (5 if tan == 5 else 1)
    if kind == "adjoint":  # forward, recomputation, and the transpose (state and adjoint in, adjoint out)
        b = n * (2 * (2 * state + cells) + 3 * state) + state
        f = n * flops * cells * (2 + 3)
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------------
# exact: the step in plain torch FP64, in definitional form
# ---------------------------------------------------------------------------

class _Exact:
    """One geometry's step F(g, T, Y; theta) with theta = (ln A, Ta, T_wall,
    u_in), all FP64.  Only fluid cells change."""

    def __init__(self, cfg, solid):
        self.cfg, self.dim = cfg, cfg["dim"]
        self.n = (cfg["nx"], cfg["ny"], cfg["nz"])
        self.C, self.w = _directions(self.dim), _weights(self.dim)
        self.Q = len(self.C)
        self.solid = solid.reshape(-1)
        nz, ny, nx = solid.shape
        idx = torch.arange(nx * ny * nz, device=DEV)
        self.xyz = [idx % nx, (idx // nx) % ny, idx // (nx * ny)]
        self.N = idx.numel()
        self._nb = {}
        self.section = float((~solid[:, :, 0]).sum())

    def neighbour(self, d, clamp=False):
        """Cell index at offset d and the non-periodic face crossed (-1: none;
        the first axis wins); clamp: index clamped at those faces."""
        key = (tuple(d), clamp)
        if key not in self._nb:
            q, face = [], torch.full((self.N,), -1, dtype=torch.int8, device=DEV)
            for a in range(3):
                v = self.xyz[a] + d[a]
                if self.cfg["bc"][2 * a] == "periodic" or a >= self.dim:
                    v = torch.remainder(v, self.n[a])
                else:
                    face = torch.where((face < 0) & (v < 0), torch.full_like(face, 2 * a), face)
                    face = torch.where((face < 0) & (v >= self.n[a]), torch.full_like(face, 2 * a + 1), face)
                    v = v.clamp(0, self.n[a] - 1)
                q.append(v)
            self._nb[key] = (q[0] + self.n[0] * (q[1] + self.n[1] * q[2]), face)
        return self._nb[key]

    # -- populations ------------------------------------------------------
    def pull(self, g, rho, th):
        cfg, dim = self.cfg, self.dim
        bc = cfg["bc"]
        Tw, u_in = th["T_wall"], th["u_in"]
        own = [sum(c[a] * g[i] for i, c in enumerate(self.C) if c[a]) * 3.0 / rho for a in range(dim)]
        out = []
        for i, c in enumerate(self.C):
            src, face = self.neighbour((-c[0], -c[1], -c[2]))
            gb = g[self.Q - 1 - i]
            v = g[i][src]
            # beyond a face `src` is the clamped boundary column: where that is
            # solid the link hits the solid
            bounce = self.solid[src]
            for f in range(2 * dim):
                t = bc[f]
                if t == "periodic" or c[f // 2] != (1 if f % 2 == 0 else -1):
                    continue
                a = f // 2
                coord = self.xyz[a] - c[a]
                at = (coord < 0) if f % 2 == 0 else (coord >= self.n[a])
                if t.startswith("wall"):
                    bounce = bounce | at
                elif t == "inlet":
                    un = u_in if f % 2 == 0 else -u_in
                    v = torch.where(at & (face == f), gb + 2.0 * self.w[i] * (c[a] * un), v)
                else:  # constant pressure
                    cu = sum(c[b] * own[b] for b in range(dim))
                    uu = sum(own[b] * own[b] for b in range(dim))
                    v = torch.where(at & (face == f), 2.0 * self.w[i] * rho * (1.5 * cu * cu - 0.5 * uu) - gb, v)
            out.append(torch.where(bounce, gb, v))
        return out

    # -- scalars along one axis -------------------------------------------
    def line(self, a, T, Y, rho, th):
        """T, Y, rho at offsets -2..2 along axis a with ghost points, and
        whether any of them is one."""
        cfg = self.cfg
        bc = cfg["bc"]
        invWk = th["invWk"]
        pts = {0: (T, Y, rho)}
        near = torch.zeros(self.N, dtype=torch.bool, device=DEV)

        def at(j):
            d = [0, 0, 0]
            d[a] = j
            return self.neighbour(tuple(d))

        c0 = torch.arange(self.N, device=DEV)
        for side in (-1, 1):
            (i1, f1), (i2, f2), (io, fo) = at(side), at(2 * side), at(-side)
            s1, s2 = self.solid[i1], self.solid[i2]
            bad1, bad2 = s1 | (f1 >= 0), s2 | (f2 >= 0)
            opp = torch.where(self.solid[io] | (fo >= 0), c0, io)
            w = torch.where(bad1, 1, torch.where(bad2, 2, 0))
            near = near | (w > 0)
            # the wall's type: the face crossed first, else solid
            face_wall = torch.where(bad1, f1 >= 0, f2 >= 0)
            src1 = torch.where(w == 1, c0, i1)
            src2 = torch.where(w == 1, opp, torch.where(w == 2, i1, i2))
            f = 2 * a + (0 if side < 0 else 1)
            for j, src, ghost in ((1, src1, w == 1), (2, src2, w > 0)):
                Tm, Ym, rm = T[src], Y[:, src], rho[src]
                Tj, Yj, rj = Tm, Ym, rm
                invW = (Ym * invWk).sum(0)

                def dirichlet(mask, TB, Tj, rj):
                    rB = th["T_in"] * th["invW_in"] / (TB * invW)
                    return torch.where(mask, 2.0 * TB - Tm, Tj), torch.where(mask, 2.0 * rB - rm, rj)

                if cfg["solid_isothermal"]:
                    Tj, rj = dirichlet(ghost & ~face_wall, th["T_wall"] if th["solid_is_wall"] else cfg["T_solid"],
                                       Tj, rj)
                if bc[f] == "wall_isothermal":
                    Tj, rj = dirichlet(ghost & face_wall, th["T_wall"], Tj, rj)
                if bc[f] == "inlet":
                    m = ghost & face_wall
                    Tj = torch.where(m, 2.0 * th["T_in"] - Tm, Tj)
                    Yj = torch.where(m, 2.0 * th["Y_in"] - Ym, Yj)
                    rj = torch.where(m, 2.0 - rm, rj)
                pts[side * j] = (Tj, Yj, rj)
        return [pts[j] for j in (-2, -1, 0, 1, 2)], near

    @staticmethod
    def d1(v):
        return (v[0] - 8.0 * v[1] + 8.0 * v[3] - v[4]) / 12.0

    @staticmethod
    def d2(v):
        return (-v[0] + 16.0 * v[1] - 30.0 * v[2] + 16.0 * v[3] - v[4]) / 12.0

    @staticmethod
    def weno(v, u, eps):
        def face(a, b, c):
            a0 = (1.0 / 3.0) / (eps + (b - a) ** 2) ** 2
            a1 = (2.0 / 3.0) / (eps + (c - b) ** 2) ** 2
            return (a0 * (1.5 * b - 0.5 * a) + a1 * 0.5 * (b + c)) / (a0 + a1)

        up = face(v[1], v[2], v[3]) - face(v[0], v[1], v[2])
        dn = face(v[4], v[3], v[2]) - face(v[3], v[2], v[1])
        return torch.where(u >= 0, up, dn)

    # -- moments ----------------------------------------------------------
    def moments(self, f, u, inverse=False):
        """Central moments sum_i f_i prod_a (c_ia - u_a)^p_a (index p + 3q +
        9r), or the populations of given central moments, axis by axis."""
        f = list(f)
        for a in (range(self.dim) if not inverse else reversed(range(self.dim))):
            s = 3 ** a
            for j in range(self.Q):
                if (j // s) % 3:
                    continue
                m, z, p = f[j], f[j + s], f[j + 2 * s]
                if not inverse:
                    f[j], f[j + s] = m + z + p, (p - m) - u[a] * (m + z + p)
                    f[j + 2 * s] = m * (1.0 + u[a]) ** 2 + z * u[a] ** 2 + p * (1.0 - u[a]) ** 2
                else:
                    r0, r1 = m, z + u[a] * m
                    r2 = p + 2.0 * u[a] * z + u[a] ** 2 * m
                    f[j], f[j + s], f[j + 2 * s] = 0.5 * (r2 - r1), r0 - r2, 0.5 * (r2 + r1)
        return f

    def products(self, k, j):
        """The part of central moment j made of lower cumulants: the sum over
        all partitions of its indices into several blocks of two or more (the
        scheme leaves first-order cumulants out)."""
        p = [j % 3, (j // 3) % 3, j // 9]
        items = [a for a in range(3) for _ in range(p[a])]
        total = 0.0
        for part in _partitions(tuple(items)):
            if len(part) < 2:
                continue
            t = 1.0
            for b in part:
                t = t * k[sum(3 ** a for a in b)]
            total = total + t
        return total

    def cumulants(self, m, inverse=False):
        k = list(m)
        for o in (4, 5, 6):  # orders below 4 are their own cumulants
            for j in range(self.Q):
                if j % 3 + (j // 3) % 3 + j // 9 == o:
                    k[j] = m[j] + self.products(m, j) if inverse else m[j] - self.products(k, j)
        return k

    def step(self, g, T, Y, th):
        cfg, dim, Q = self.cfg, self.dim, self.Q
        invWk = th["invWk"]
        invW = (Y * invWk).sum(0)
        rho = th["T_in"] * th["invW_in"] / (T * invW)
        f = self.pull(g, rho, th)
        u = [3.0 * sum(c[a] * f[i] for i, c in enumerate(self.C) if c[a]) / rho for a in range(dim)]
        alpha = cfg["nu"] / cfg["Pr"]
        D = torch.tensor([alpha / le for le in cfg["Le"]], dtype=torch.float64, device=DEV)[:, None]
        Wk = 1.0 / invWk
        convT = diffT = 0.0
        convY = diffY = 0.0
        grad = []
        for a in range(dim):
            pts, near = self.line(a, T, Y, rho, th)
            Tl, Yl, rl = [p[0] for p in pts], [p[1] for p in pts], [p[2] for p in pts]
            iW = [(y * invWk).sum(0) for y in Yl]
            drho = self.d1(rl)
            grad.append(drho)
            dr = drho / rho
            c2 = 0.5 * (Tl[3] - Tl[1])
            convT = convT + u[a] * torch.where(near, c2, self.weno(Tl, u[a], th["eps"] * th["T_in"] ** 2))
            diffT = diffT + alpha * (self.d2(Tl) + dr * self.d1(Tl))
            L = torch.where(near, 0.5 * (Yl[3] - Yl[1]), self.weno(Yl, u[a], th["eps"]))
            convY = convY + u[a] * (L - Y * L.sum(0))
            Xl = [y * invWk / v for y, v in zip(Yl, iW)]
            dX, d2X, dY = self.d1(Xl), self.d2(Xl), self.d1(Yl)
            m = D * Wk * invW * dX
            dm = D * Wk * (invW * d2X + self.d1(iW) * dX)
            M, dM = m.sum(0), dm.sum(0)
            diffY = diffY + dm - dY * M - Y * dM + (m - Y * M) * dr
        q = th["A"] * Y[cfg["fuel"]].clamp(min=0) * Y[cfg["oxidiser"]].clamp(min=0) * torch.exp(-th["Ta"] / T)
        yF = -cfg["nu_stoich"][cfg["fuel"]] * cfg["W"][cfg["fuel"]]
        yld = torch.tensor([n * w / yF for n, w in zip(cfg["nu_stoich"], cfg["W"])], dtype=torch.float64,
                           device=DEV)[:, None]
        DT = diffT + cfg["Q"] / cfg["cp"] * q
        DY = diffY + yld * q
        Lam = DT / T + (DY * invWk).sum(0) / invW
        Tn, Yn = T + DT - convT, Y + DY - convY
        # collision
        rc = rho * CS2
        Ph = sum(f) + 0.5 * rc * Lam
        uu = sum(v * v for v in u)
        xi, pre, eq = [], [], []
        for i, c in enumerate(self.C):
            cu = sum(c[a] * u[a] for a in range(dim))
            r = self.w[i] * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu)
            x = CS2 * (r - self.w[i]) * sum((c[a] - u[a]) * grad[a] for a in range(dim)) + self.w[i] * rc * Lam
            xi.append(x)
            pre.append((f[i] + 0.5 * x) / rc)
            eq.append(self.w[i] * (Ph / rc - 1.0) + r)
        k = self.cumulants(self.moments(pre, u))
        ke = self.cumulants(self.moments(eq, u))
        ws = 1.0 / (3.0 * cfg["nu"] + 0.5)
        wb = cfg["omega_bulk"] if cfg["omega_bulk"] > 0 else ws
        new = list(k)
        second = [2 * 3 ** a for a in range(dim)]
        for j in range(Q):
            o = j % 3 + (j // 3) % 3 + j // 9
            if o >= 3:
                new[j] = ke[j] + (1.0 - cfg["omega_hi"]) * (k[j] - ke[j])
            elif o == 2:
                new[j] = ke[j] + (1.0 - ws) * (k[j] - ke[j])
        tr = sum(k[j] - ke[j] for j in second)
        for j in second:  # the trace relaxes at its own rate
            new[j] = new[j] + (ws - wb) * tr / dim
        out = self.moments(self.cumulants(new, inverse=True), u, inverse=True)
        gn = [rc * out[i] + 0.5 * xi[i] for i in range(Q)]
        s = self.solid
        return (torch.stack([torch.where(s, g[i], gn[i]) for i in range(Q)]), torch.where(s, T, Tn),
                torch.where(s, Y, Yn))


_PARTS = {}


def _partitions(items):
    """All set partitions of `items` (with repetition) into blocks of two or more."""
    if items in _PARTS:
        return _PARTS[items]

    def rec(rest):
        if not rest:
            return [[]]
        head, tail = rest[0], rest[1:]
        found = []
        for mask in range(1 << len(tail)):
            block = [head] + [t for b, t in enumerate(tail) if mask >> b & 1]
            if len(block) < 2:
                continue
            left = [t for b, t in enumerate(tail) if not mask >> b & 1]
            found += [[block] + p for p in rec(left)]
        return found

    _PARTS[items] = rec(list(items))
    return _PARTS[items]


def _theta(cfg):
    """theta = (ln A, Ta, T_wall, u_in) of a configuration; T_wall moves the
    isothermal walls and the isothermal solid together."""
    walls = [cfg["T_wall"][f] for f, b in enumerate(cfg["bc"]) if b == "wall_isothermal"]
    return torch.tensor([math.log(cfg["A"]), cfg["Ta"], walls[0] if walls else cfg["T_solid"], cfg["u_in"]],
                        dtype=torch.float64, device=DEV)


def _params(cfg, theta, u_in=None):
    f64 = dict(dtype=torch.float64, device=DEV)
    return dict(A=torch.exp(theta[0]) * cfg["dt"], Ta=theta[1], T_wall=theta[2],
                u_in=theta[3] if u_in is None else u_in, solid_is_wall=bool(cfg["solid_isothermal"]),
                T_in=cfg["T_in"], eps=cfg["weno_eps"], Y_in=torch.tensor(cfg["Y_in"], **f64)[:, None],
                invWk=1.0 / torch.tensor(cfg["W"], **f64)[:, None],
                invW_in=sum(a / b for a, b in zip(cfg["Y_in"], cfg["W"])))


def _rate(cfg, th, T, Y):
    rho = th["T_in"] * th["invW_in"] / (T * (Y * th["invWk"]).sum(0))
    q = th["A"] * Y[cfg["fuel"]].clamp(min=0) * Y[cfg["oxidiser"]].clamp(min=0) * torch.exp(-th["Ta"] / T)
    return rho, q, rho * cfg["Q"] / cfg["cp"] * q


def _diag(cfg, E, th, T, Y, rows):
    """The observables of rows y0 <= y < y1 in the order of DIAG."""
    nz, ny, nx = E.n[2], E.n[1], E.n[0]
    rho, q, h = _rate(cfg, th, T, Y)
    sl = (slice(None), slice(*rows), slice(None))
    box = lambda v: v.reshape(nz, ny, nx)[sl]  # noqa: E731
    fl = ~box(E.solid)
    r, qq, hh, yf, t = box(rho), box(q), box(h), box(Y[cfg["fuel"]]), box(T)
    zero = torch.zeros_like(r)
    total = lambda v: float(torch.where(fl, v, zero).sum())  # noqa: E731
    mid = (rows[0] + rows[1]) // 2
    line = torch.where(~E.solid.reshape(nz, ny, nx)[nz // 2 if nz > 1 else 0, mid],
                       h.reshape(nz, ny, nx)[nz // 2 if nz > 1 else 0, mid], torch.full((nx,), -math.inf, device=DEV,
                                                                                       dtype=torch.float64))
    best = line.max()
    x = float(torch.nonzero(line == best)[0]) if bool(torch.isfinite(best)) else -1.0
    return [total(yf) / (cfg["Y_in"][cfg["fuel"]] * float(fl[:, :, 0].sum())), total(r), total(hh), total(r * qq),
            float(t[fl].max()), x, 0.0, float(fl.sum())]


def _front(cfg, E, th, T, Y, rows):
    nx, ny = E.n[0], E.n[1]
    _, _, h = _rate(cfg, th, T, Y)
    band = h.reshape(ny, nx)[rows[0]:rows[1]]
    peak, at = band.max(0)
    first = (band == peak).to(torch.int64).argmax(0).to(torch.float64)
    return torch.stack([peak, torch.minimum(first + 0.5, (rows[1] - rows[0]) - 0.5 - first)])


def exact(case, seed):
    cfg, solid, band, rows = _geometry(case)
    g, T, Y = _fields(cfg, solid, band, seed)
    dt = STORE[case["precision"]]
    g, T, Y = (v.to(dt).to(torch.float64) for v in (g, T, Y))
    E = _Exact(cfg, solid)
    theta = _theta(cfg)
    n, kind = case["steps"], case["kind"]
    fuel = cfg["fuel"]
    fluid = ~E.solid
    xf_scale = 1.0 / (cfg["Y_in"][fuel] * E.section)

    def advance(theta, steps, g, T, Y, u_in=None):
        th = _params(cfg, theta, u_in)
        for _ in range(steps):
            g, T, Y = E.step(g, T, Y, th)
        return g, T, Y

    out = {}
    if kind == "hold":
        ctl = dict(target=None, last=None, u=cfg["u_in"])
        xf = lambda Y: float(Y[fuel][fluid].sum()) * xf_scale  # noqa: E731
        ctl["target"] = xf(Y) + 5.0
        hist, done = [], 0
        while done < n:
            m = min(case["every"], n - done)
            g, T, Y = advance(theta, m, g, T, Y, ctl["u"])
            done += m
            x = xf(Y)
            err = ctl["target"] - x
            de = 0.0 if ctl["last"] is None else err - ctl["last"]
            ctl["last"] = err
            ctl["u"] = min(max(ctl["u"] + 1e-3 * de + 2e-5 * err, 0.0), 0.1)
            hist.append((x, ctl["u"]))
        out["history"] = np.array(hist)
    elif kind == "adjoint" or case["precision"] == "tangent":
        th0 = theta.clone().requires_grad_(True)
        seg = max(1, int(math.sqrt(n)))
        st, done = (g, T, Y), 0
        while done < n:
            m = min(seg, n - done)
            st = torch.utils.checkpoint.checkpoint(lambda t, a, b, c, m=m: advance(t, m, a, b, c), th0, *st,
                                                   use_reentrant=False)
            done += m
        J = cfg["dx"] * st[2][fuel][fluid].sum() * xf_scale
        (grad,) = torch.autograd.grad(J, th0)
        out["J"], out["grad"] = float(J.detach()), grad.cpu().numpy()
        st = tuple(v.detach() for v in st)
        if kind == "adjoint":
            g, T, Y = st
        else:
            g, T, Y = _dual(advance, theta, n, g, T, Y)
    elif case["precision"] == "tangent_mixed":
        g, T, Y = _dual(advance, theta, n, g, T, Y)
    else:
        g, T, Y = advance(theta, n, g, T, Y)
    th = _params(cfg, theta)
    if kind == "batch" and case["precision"] == "fp64":
        out["diag"] = np.array([_diag(cfg, E, th, T, Y, r) for r in rows])
        out["front"] = torch.stack([_front(cfg, E, th, T, Y, r) for r in rows]).cpu().numpy()
    if kind == "packing" and case["precision"] == "fp64":
        d = _diag(cfg, E, th, T, Y, (0, cfg["ny"]))
        out["flame"] = np.array([d[0] * cfg["dx"], d[1], d[2]])
    out["state"] = {"g": g, "T": T, "Y": Y}
    return out


def _dual(advance, theta, n, g, T, Y):
    """The state after n steps and its derivatives with respect to theta,
    stacked last (value, d/d ln A, d/d Ta, d/d T_wall, d/d u_in)."""
    parts = None
    for k in range(4):
        e = torch.zeros_like(theta)
        e[k] = 1.0
        val, der = torch.func.jvp(lambda t: advance(t, n, g, T, Y), (theta,), (e,))
        parts = [[v] for v in val] if parts is None else parts
        for p, d in zip(parts, der):
            p.append(d)
    return tuple(torch.stack(p, dim=-1) for p in parts)
