"""The work a user of the P-TRT lattice Boltzmann library has it do, as timed cases.

A case is a dict of plain values:

  lattice, nx, ny, nz, storage, layout, collision   as ``Lattice`` takes them
  flow      "shear" (double shear layer), "vortex" (Taylor-Green, 2-D or 3-D),
            "channel" (walls at both y ends, body force), "body" (solid square
            in a periodic forced lattice) or "cylinder" (the same square between
            a moving-wall inlet and a constant-density outlet)
  nu, inv_tau_minus                                 the two relaxation rates
  steps     time steps of one pass (even, so that the state is back in ``pop_a``)
  call      what a pass is:
            "solve"   init_equilibrium from device fields, step, macros
            "march"   step, diagnostics (the loop of a running simulation)
            "advance" step alone (between two outputs)
            "drag"    step, momentum_exchange (a body's force history)
            "batch"   Batch.step of many uneven lattices
            "host"    init_equilibrium and macros through pinned host buffers
            "restart" set_populations, step, populations
  tune      the program autotunes the lattice (or the batch) once before it starts
  lattices  lattices of a batch; nx and ny are then their largest extents

States are returned whole, in the storage type of the lattice: the population
planes that the program itself owns, without the padding of their rows.
"""
import math
import random

import numpy as np
import torch

from paper_2602_06686_gb300 import Batch, Lattice

KAPPA, DELTA = 80.0, 0.05
DTYPES = {"F64": torch.float64, "F32": torch.float32, "F16": torch.float16,
          "BF16": torch.bfloat16}
ESIZE = {"F64": 8, "F32": 4, "F16": 2, "BF16": 2}
Q_OF = {"D2Q9": 9, "D3Q19": 19, "D3Q27": 27}
# floating point operations of one P-TRT node update, moments to relaxation
FLOPS = {"D2Q9": 130, "D3Q19": 300, "D3Q27": 450}


def _case(name, lattice, nx, ny, nz, storage, flow, nu, steps, call, layout="AB",
          collision="P_TRT", inv_tau_minus=1.6, tune=False, lattices=0):
    return {"name": name, "lattice": lattice, "nx": nx, "ny": ny, "nz": nz, "storage": storage,
            "flow": flow, "nu": nu, "steps": steps, "call": call, "layout": layout,
            "collision": collision, "inv_tau_minus": inv_tau_minus, "tune": tune,
            "lattices": lattices}


def listed():
    return [
        # A whole small FP64 validation run: start, march, read the fields.
        _case("solve_d2q9_f64_64", "D2Q9", 64, 64, 1, "F64", "vortex", 0.01, 100, "solve"),
        # A parameter study's lattice of ordinary size, diagnosed as it runs.
        _case("march_d2q9_f32_1024", "D2Q9", 1024, 1024, 1, "F32", "shear", 0.01024, 100,
              "march"),
        # The benchmark of the library: the large shear layer, diagnosed as it runs.
        _case("march_d2q9_f32_4096", "D2Q9", 4096, 4096, 1, "F32", "shear", 0.004096, 50, "march",
              tune=True),
        # Reduced-precision storage on a lattice of no special extent.
        _case("advance_d2q9_f16_2250x1410", "D2Q9", 2250, 1410, 1, "F16", "shear", 0.0141, 50,
              "advance", tune=True),
        # The square cylinder array: solid mask, body force, force history.
        _case("drag_d2q9_f32_body", "D2Q9", 2048, 1024, 1, "F32", "body", 0.5, 50, "drag",
              tune=True),
        # The drag benchmark in FP64: solid square between inlet and outlet.
        _case("drag_d2q9_f64_cylinder", "D2Q9", 1050, 1050, 1, "F64", "cylinder", 0.3, 20,
              "drag"),
        # The 3-D Taylor-Green vortex at its full size.
        _case("march_d3q19_f32_384", "D3Q19", 384, 384, 384, "F32", "vortex", 0.0019, 10, "march",
              tune=True),
        # FP64 in three dimensions: the reference run of a precision study.
        _case("march_d3q19_f64_96", "D3Q19", 96, 96, 96, "F64", "vortex", 0.01, 10, "march"),
        # The walled, force-driven channel with 16-bit storage.
        _case("advance_d3q19_f16_channel", "D3Q19", 512, 64, 512, "F16", "channel", 0.1, 10,
              "advance", inv_tau_minus=1.1, tune=True),
        # Half the memory: in place, on an extent that is no multiple of anything.
        _case("restart_d3q19_f32_aa", "D3Q19", 150, 131, 117, "F32", "vortex", 0.01, 10,
              "restart", layout="AA"),
        # The 27-velocity lattice, fields exchanged with the host around the steps.
        _case("host_d3q27_f32_192", "D3Q27", 192, 192, 192, "F32", "vortex", 0.01, 20, "host"),
        # A sweep over Reynolds numbers: uneven lattices stepped together.
        _case("batch_d2q9_f32_256", "D2Q9", 1024, 1024, 1, "F32", "shear", 0.01, 20, "batch",
              tune=True, lattices=256),
    ]


def _loguniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng: random.Random):
    call = rng.choice(["solve", "march", "march", "advance", "advance", "drag", "restart", "host",
                       "batch"])
    if call == "batch":
        return _draw_batch(rng)
    lattice = "D2Q9" if call == "drag" else rng.choice(["D2Q9", "D2Q9", "D3Q19", "D3Q19", "D3Q27"])
    storage = rng.choice(["F32", "F32", "F16", "F64", "BF16"])
    if call in ("march", "drag") and storage in ("F16", "BF16"):
        storage = "F32"  # diagnostics are followed in FP32 and FP64
    steps = 2 * int(round(_loguniform(rng, 2, 50)))
    # nodes of a lattice: the work of a pass stays below the largest listed one
    top = 4096.0 ** 2 if lattice == "D2Q9" else (384.0 ** 3 if lattice == "D3Q19" else 256.0 ** 3)
    per_step = 1.6e10 if storage != "F64" else 1.5e9
    if call in ("solve", "host", "restart"):
        top = min(top, 8e6)
    top = min(top, per_step / (Q_OF[lattice] * ESIZE[storage] * steps))
    nodes = _loguniform(rng, 64.0 ** 2 if lattice == "D2Q9" else 32.0 ** 3, max(top, 5e4))

    def side(mean):
        n = max(16, int(round(mean * rng.uniform(0.75, 1.3))))
        return n if rng.random() < 0.4 else max(16, (n + 8) // 16 * 16)

    if lattice == "D2Q9":
        nx, ny, nz = side(nodes ** 0.5), side(nodes ** 0.5), 1
    else:
        nx, ny, nz = (side(nodes ** (1.0 / 3.0)) for _ in range(3))
    flow = "vortex"
    if call == "drag":
        flow = rng.choice(["body", "cylinder"])
    elif lattice == "D2Q9" and min(nx, ny) >= 256 and rng.random() < 0.5:
        flow = "shear"
    elif rng.random() < 0.3:
        flow = "channel"
    layout = "AA" if flow not in ("body", "cylinder") and rng.random() < 0.2 else "AB"
    collision = rng.choice(["P_TRT", "P_TRT", "P_TRT", "TRT"] +
                           (["TRT_RLB"] if lattice != "D3Q27" else []))
    nu = 0.1 if flow == "channel" else _loguniform(rng, 0.01, 0.2)
    c = _case("", lattice, nx, ny, nz, storage, flow, round(nu, 5), steps, call, layout, collision,
              1.6 if flow != "channel" else 1.1, rng.random() < 0.5)
    del c["name"]
    return c


def _draw_batch(rng):
    storage = rng.choice(["F32", "F32", "F16"])
    c = _case("", "D2Q9", rng.randint(128, 1024), rng.randint(128, 1024), 1, storage, "shear",
              0.01, 2 * rng.randint(3, 10), "batch", lattices=int(_loguniform(rng, 8, 200)))
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _rng(seed):
    return np.random.default_rng(seed)


def _solid(case):
    """A centred solid square: a 32nd (array) or a 50th (drag benchmark) of the
    lattice's longer side."""
    if case["flow"] not in ("body", "cylinder"):
        return None
    nx, ny = case["nx"], case["ny"]
    side = max(3, max(nx, ny) // (32 if case["flow"] == "body" else 50))
    m = np.zeros((1, ny, nx), dtype=np.uint8)
    x0, y0 = (nx - side) // 2, (ny - side) // 2
    m[0, y0:y0 + side, x0:x0 + side] = 1
    return m


def _force(case):
    D = 2 if case["lattice"] == "D2Q9" else 3
    if case["flow"] == "channel":
        return (8.0 * case["nu"] * 0.05 / case["ny"] ** 2,) + (0.0,) * 2
    if case["flow"] == "body":
        return (1e-6, 2e-7, 0.0)[:D] + (0.0,) * (3 - D)
    return (0.0, 0.0, 0.0)


def _periodic(case):
    if case["flow"] == "channel":
        return (1, 0, 1)
    if case["flow"] == "cylinder":
        return (0, 1, 1)
    return (1, 1, 1)


def _inlet(case):
    return (0.02, 1.0)  # inlet velocity, outlet density of the drag benchmark


def _fields(nx, ny, nz, D, flow, r, device, solid=None):
    """Seeded smooth FP64 (rho, u): phases, amplitude and a slow mean stream
    (the frame the flow is seen from) are drawn from `r`."""
    f64 = torch.float64
    px, py, pz = r.uniform(0, 2 * math.pi, 3)
    amp = r.uniform(0.04, 0.05)
    mean = r.uniform(0.005, 0.015, 3)
    X = (torch.arange(nx, dtype=f64, device=device) * (2 * math.pi / nx) + px).view(1, 1, nx)
    Y = (torch.arange(ny, dtype=f64, device=device) * (2 * math.pi / ny) + py).view(1, ny, 1)
    Z = (torch.arange(nz, dtype=f64, device=device) * (2 * math.pi / nz) + pz).view(nz, 1, 1)
    u = torch.empty((D, nz, ny, nx), dtype=f64, device=device)
    if flow == "shear":
        y = torch.arange(ny, dtype=f64, device=device).view(1, ny, 1) / ny
        U0 = 2.0 * amp
        prof = torch.where(y <= 0.5, U0 * torch.tanh(KAPPA * (y - 0.25)),
                           U0 * torch.tanh(KAPPA * (0.75 - y)))
        u[0] = prof + mean[0]
        u[1] = DELTA * U0 * torch.sin(X) + mean[1]
        rho = torch.ones((nz, ny, nx), dtype=f64, device=device)
    elif flow == "channel":
        y = (torch.arange(ny, dtype=f64, device=device).view(1, ny, 1) + 0.5) / ny
        u[0] = 4 * amp * y * (1 - y) * (1.0 + 0.05 * torch.sin(X) * torch.cos(Z))
        u[1] = 0.002 * torch.sin(math.pi * y) * torch.cos(X)
        if D == 3:
            u[2] = 0.004 * torch.sin(math.pi * y) * torch.sin(X + Z) + mean[2] * y * (1 - y)
        rho = 1.0 + 0.001 * torch.cos(X + Z).expand(nz, ny, nx)
    elif flow in ("body", "cylinder"):
        scale = 0.1 if flow == "body" else 0.02 / 0.05
        base = 0.02 if flow == "cylinder" else mean[0]
        u[0] = base + scale * 0.02 * torch.sin(Y) * torch.cos(X)
        u[1] = scale * 0.02 * torch.cos(Y) * torch.sin(X) + (0.0 if flow == "cylinder" else 0.002)
        rho = 1.0 + 0.0005 * torch.cos(X + Y).expand(nz, ny, nx)
    else:
        cz = torch.cos(Z) if D == 3 else torch.ones_like(Z)
        u[0] = amp * torch.sin(X) * torch.cos(Y) * cz + mean[0]
        u[1] = -amp * torch.cos(X) * torch.sin(Y) * cz + mean[1]
        if D == 3:
            u[2] = mean[2]
            p = amp * amp * 3.0 / 16.0 * (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2)
        else:
            p = amp * amp * 0.75 * (torch.cos(2 * X) + torch.cos(2 * Y))
        rho = 1.0 + p
    if solid is not None:
        u *= torch.as_tensor(solid == 0, device=device)
    return rho.contiguous(), u


def _batch_members(case, r):
    """Uneven extents (64 to nx, 64 to ny) and viscosities of a sweep's lattices."""
    out = []
    for _ in range(case["lattices"]):
        out.append((int(r.integers(64, case["nx"] + 1)), int(r.integers(64, case["ny"] + 1)),
                    float(10.0 ** r.uniform(-2.5, -1.0))))
    return out


def _kw(case):
    return dict(lattice=case["lattice"], nx=case["nx"], ny=case["ny"], nz=case["nz"],
                nu=case["nu"], tau_minus=1.0 / case["inv_tau_minus"], collision=case["collision"],
                force=_force(case), periodic=_periodic(case), storage=case["storage"],
                layout=case["layout"])


def _planes(g, buf, storage):
    """The population planes [Q, nz, ny, nx] in a buffer of lattice g (a view)."""
    t = buf.view(DTYPES[storage])
    per = 16 // ESIZE[storage]
    pitch = (g.p.nx + per - 1) // per * per
    plane = t.numel() // g.Q
    cells = pitch * g.p.ny * g.p.nz
    return t.view(g.Q, plane)[:, :cells].view(g.Q, g.p.nz, g.p.ny, pitch)[..., :g.p.nx]


def prepare(case, seed):
    dev = torch.device("cuda")
    D = 2 if case["lattice"] == "D2Q9" else 3
    st = {"case": case}
    if case["call"] == "batch":
        members = _batch_members(case, _rng(1000 + case["lattices"]))
        b = Batch([dict(lattice="D2Q9", nx=nx, ny=ny, nu=nu, tau_minus=1.0 / case["inv_tau_minus"],
                        collision=case["collision"], storage=case["storage"])
                   for nx, ny, nu in members])
        b.pop_a.zero_()
        b.pop_b.zero_()
        r = _rng(seed)
        inputs = [_fields(nx, ny, 1, 2, "shear", r, dev) for nx, ny, _ in members]
        for v, (rho, u) in zip(b.views, inputs):
            v.init_equilibrium(rho, u)
        if case["tune"]:
            b.autotune(steps=4)  # takes real steps: the sweep starts afresh
            for v, (rho, u) in zip(b.views, inputs):
                v.init_equilibrium(rho, u)
        st["b"] = b
        return st
    solid = _solid(case)
    rho, u = _fields(case["nx"], case["ny"], case["nz"], D, case["flow"], _rng(seed), dev, solid)
    g = Lattice(solid=solid, **_kw(case))
    g.pop_a.zero_()
    if g.pop_b is not None:
        g.pop_b.zero_()
    if case["flow"] == "cylinder":
        g.set_open_boundaries(*_inlet(case))
    g.init_equilibrium(rho, u)
    if case["tune"]:
        g.autotune(reps=3, report=False)
        g.init_equilibrium(rho, u)
    st["g"] = g
    if case["call"] == "solve":
        st["rho"], st["u"] = rho, u
    elif case["call"] == "host":
        st["rho"], st["u"] = rho.cpu().pin_memory(), u.cpu().pin_memory()
        st["rho_out"] = torch.empty(rho.shape, dtype=torch.float64, pin_memory=True)
        st["u_out"] = torch.empty(u.shape, dtype=torch.float64, pin_memory=True)
    elif case["call"] == "restart":
        st["f"] = g.populations()
    return st


def run(state):
    case = state["case"]
    n = case["steps"]
    call = case["call"]
    if call == "batch":
        b = state["b"]
        b.step(n)
        return {"state": b.pop_a.view(DTYPES[case["storage"]])}
    g = state["g"]
    if call == "solve":
        g.init_equilibrium(state["rho"], state["u"])
        g.step(n)
        rho, u = g.macros()
        return {"rho": rho, "u": u}
    if call == "host":
        g.init_equilibrium_host_ptr(state["rho"].data_ptr(), state["u"].data_ptr())
        g.step(n)
        g.macros_host_ptr(state["rho_out"].data_ptr(), state["u_out"].data_ptr())
        return {"state": _planes(g, g.pop_a, case["storage"]), "rho": state["rho_out"],
                "u": state["u_out"]}
    if call == "restart":
        g.set_populations(state["f"])
        g.step(n)
        return {"f": g.populations()}
    g.step(n)
    out = {"state": _planes(g, g.pop_a, case["storage"])}
    if call == "march":
        d = g.diagnostics()
        out.update(mass=d["mass"], momentum=d["momentum"], kinetic_energy=d["kinetic_energy"],
                   enstrophy=d["enstrophy"], nan_flag=d["nan_flag"], step=d["step"])
    elif call == "drag":
        out["force"] = g.momentum_exchange()
    return out


def work(case):
    """One pass: the state read once and written once (however many steps it
    advances), the mask and the fields that enter or leave, and every step's
    arithmetic."""
    Q, e = Q_OF[case["lattice"]], ESIZE[case["storage"]]
    D = 2 if case["lattice"] == "D2Q9" else 3
    if case["call"] == "batch":
        n = sum(nx * ny for nx, ny, _ in _batch_members(case, _rng(1000 + case["lattices"])))
    else:
        n = case["nx"] * case["ny"] * case["nz"]
    b = 2 * Q * e * n
    if case["flow"] in ("body", "cylinder"):
        b += n
    if case["call"] in ("solve", "host"):
        b = 2 * (1 + D) * 8 * n
    elif case["call"] == "restart":
        b = 2 * Q * 8 * n
    return {"bytes": b, "flops": FLOPS[case["lattice"]] * n * case["steps"]}


# ------------------------------------------------------------------ exact
def _velocities(lattice):
    """Velocities, weights and opposites in the order of the library."""
    if lattice == "D2Q9":
        e = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0),
             (-1, -1, 0), (1, -1, 0)]
    else:
        e = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
        for a, b in ((0, 1), (0, 2), (1, 2)):
            for sa, sb in ((1, 1), (-1, -1), (1, -1), (-1, 1)):
                v = [0, 0, 0]
                v[a], v[b] = sa, sb
                e.append(tuple(v))
        if lattice == "D3Q27":
            for v in ((1, 1, 1), (1, 1, -1), (1, -1, 1), (-1, 1, 1)):
                e += [v, tuple(-c for c in v)]
    n2 = [sum(c * c for c in v) for v in e]
    w = {"D2Q9": (4 / 9, 1 / 9, 1 / 36), "D3Q19": (1 / 3, 1 / 18, 1 / 36),
         "D3Q27": (8 / 27, 2 / 27, 1 / 54, 1 / 216)}[lattice]
    opp = [e.index(tuple(-c for c in v)) for v in e]
    return e, [w[k] for k in n2], opp


class _Exact:
    """The scheme in plain FP64 torch, on shifted populations g_i = f_i - w_i."""

    def __init__(self, case, shape, nu, solid, device):
        self.case, self.shape = case, shape
        self.e, self.w, self.opp = _velocities(case["lattice"])
        self.D = 2 if case["lattice"] == "D2Q9" else 3
        self.F = _force(case) if case["call"] != "batch" else (0.0, 0.0, 0.0)
        self.per = _periodic(case)
        self.wp = 1.0 / (0.5 + 3.0 * nu)
        self.wm = case["inv_tau_minus"]
        self.solid = None if solid is None else torch.as_tensor(solid != 0, device=device)

    def macros(self, g):
        drho = sum(g)
        j = [sum(c[a] * gi for c, gi in zip(self.e, g) if c[a]) for a in range(self.D)]
        rho = 1.0 + drho
        return drho, rho, [(j[a] + 0.5 * self.F[a]) / rho for a in range(self.D)]

    def _parts(self, i, drho, rho, u, usq):
        """Symmetric and antisymmetric part of the shifted equilibrium of i."""
        eu = sum(c * ua for c, ua in zip(self.e[i], u) if c)
        w = self.w[i]
        return (w * (drho + rho * (4.5 * eu * eu - 1.5 * usq)),
                w * rho * eu * (3.0 + 4.5 * (eu * eu - usq)), eu)

    def equilibrium(self, rho, u):
        usq = sum(c * c for c in u)
        g = []
        for i in range(len(self.e)):
            s, a, _ = self._parts(i, rho - 1.0, rho, u, usq)
            g.append(s + a)
        return self._clear(g)

    def _clear(self, g):
        if self.solid is not None:
            for gi in g:
                gi.masked_fill_(self.solid, 0.0)
        return g

    def collide(self, g):
        D, e, w = self.D, self.e, self.w
        drho, rho, u = self.macros(g)
        usq = sum(c * c for c in u)
        uF = sum(ua * f for ua, f in zip(u, self.F) if f)
        hg = 1.0 - 0.5 * self.wp
        A2 = {}  # second moments of the non-equilibrium
        for a in range(D):
            for b in range(a, D):
                m = sum(c[a] * c[b] * gi for c, gi in zip(e, g) if c[a] * c[b])
                A2[a, b] = m - rho * u[a] * u[b] - (drho / 3.0 if a == b else 0.0)
        out = [None] * len(e)
        for i in range(len(e)):
            k = self.opp[i]
            if k < i:
                continue
            fs, fa, eu = self._parts(i, drho, rho, u, usq)
            if self.case["collision"] == "TRT":
                r2 = 0.5 * (g[i] + g[k]) - fs
            else:  # purified: only the second Hermite moments of the non-equilibrium are left
                r2 = 0.0
                for (a, b), m in A2.items():
                    h = e[i][a] * e[i][b] - (1.0 / 3.0 if a == b else 0.0)
                    if h:
                        r2 = r2 + (4.5 * w[i] * h * (1.0 if a == b else 2.0)) * m
            eF = sum(c * f for c, f in zip(e[i], self.F))
            sym = fs + (1.0 - self.wp) * r2
            anti = fa + (1.0 - self.wm) * (0.5 * (g[i] - g[k]) - fa)
            if any(self.F):
                sym = sym + hg * w[i] * (9.0 * eF * eu - 3.0 * uF)
                anti = anti + 1.5 * w[i] * eF * (2.0 - self.wm)
            out[i] = sym + anti
            if k != i:
                out[k] = sym - anti
        return self._clear(out)

    def stream(self, f):
        """Pull: the population of the upstream node, or the node's own opposite
        one where that is solid or beyond a wall."""
        g = []
        for i, c in enumerate(self.e):
            v = f[i]
            back = None
            for a, dim in ((0, 2), (1, 1), (2, 0)):
                if c[a]:
                    v = torch.roll(v, c[a], dim)
            if self.solid is not None:
                back = self.solid
                for a, dim in ((0, 2), (1, 1), (2, 0)):
                    if c[a]:
                        back = torch.roll(back, c[a], dim)
            for a, dim in ((0, 2), (1, 1), (2, 0)):
                if c[a] and not self.per[a]:
                    n = self.shape[dim]
                    line = torch.zeros(n, dtype=torch.bool, device=v.device)
                    line[0 if c[a] > 0 else n - 1] = True
                    line = line.view([n if d == dim else 1 for d in range(3)])
                    back = line.expand(self.shape) if back is None else back | line
            if back is not None:
                v = torch.where(back, f[self.opp[i]], v)
            g.append(v)
        if self.case["flow"] == "cylinder":
            self._open(g)
        return self._clear(g)

    def _open(self, g):
        u_in, rho_out = _inlet(self.case)
        e = self.e
        for i, c in enumerate(e):
            if c[0] == 1:
                g[i][..., 0] += 6.0 * self.w[i] * u_in
        s0 = sum(g[i][..., -1] for i, c in enumerate(e) if c[0] == 0)
        sp = sum(g[i][..., -1] for i, c in enumerate(e) if c[0] == 1)
        up = g[e.index((0, 1, 0))][..., -1].clone()
        down = g[e.index((0, -1, 0))][..., -1].clone()
        ux = (s0 + 2.0 * sp + 1.0 - rho_out) / rho_out
        for i, c in enumerate(e):
            if c[0] == -1:
                g[i][..., -1] = g[self.opp[i]][..., -1] - 6.0 * self.w[i] * rho_out * ux \
                    - 0.5 * c[1] * (up - down)

    def drag(self, g):
        f = self.collide(g)
        out = [0.0, 0.0, 0.0]
        for i, c in enumerate(self.e):
            if not any(c):
                continue
            ahead = self.solid
            for a, dim in ((0, 2), (1, 1), (2, 0)):
                if c[a]:
                    ahead = torch.roll(ahead, -c[a], dim)
            link = ahead & ~self.solid
            s = float((2.0 * (f[i] + self.w[i]))[link].sum())
            for a in range(3):
                out[a] += c[a] * s
        return np.array(out)

    def diagnostics(self, g):
        drho, rho, u = self.macros(g)
        usq = sum(c * c for c in u)

        def d(a, b):  # central difference of u_a along axis b (walls: u = 0 beyond)
            dim = 2 - b
            n = self.shape[dim]
            p, m = torch.roll(u[a], -1, dim), torch.roll(u[a], 1, dim)
            if not self.per[b]:
                p.select(dim, n - 1).zero_()
                m.select(dim, 0).zero_()
            return 0.5 * (p - m)

        if self.D == 2:
            curl = (d(1, 0) - d(0, 1)) ** 2
        else:
            curl = (d(2, 1) - d(1, 2)) ** 2 + (d(0, 2) - d(2, 0)) ** 2 + (d(1, 0) - d(0, 1)) ** 2
        mom = [float((rho * c).sum()) for c in u] + [0.0] * (3 - self.D)
        return {"mass": float(rho.sum()), "momentum": np.array(mom),
                "kinetic_energy": float((0.5 * rho * usq).sum()),
                "enstrophy": float(0.5 * curl.sum()), "nan_flag": None, "step": None}


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    D = 2 if case["lattice"] == "D2Q9" else 3
    n = case["steps"]
    if case["call"] == "batch":
        return _exact_batch(case, seed, dev)
    solid = _solid(case)
    shape = (case["nz"], case["ny"], case["nx"])
    rho, u = _fields(case["nx"], case["ny"], case["nz"], D, case["flow"], _rng(seed), dev, solid)
    X = _Exact(case, shape, case["nu"], solid, dev)
    g = X.equilibrium(rho, [u[a] for a in range(D)])
    del rho, u
    f = g
    for s in range(n):
        f = X.collide(g)
        del g
        g = X.stream(f) if s + 1 < n or case["call"] != "advance" or case["layout"] == "AA" else None
    call = case["call"]
    if call in ("solve", "host"):
        _, rho, u = X.macros(g)
        u = torch.stack(u)
        if call == "solve":
            return {"rho": rho, "u": u}
        return {"state": torch.stack(f if case["layout"] == "AB" else g), "rho": rho.cpu(),
                "u": u.cpu()}
    if call == "restart":
        w = torch.tensor(X.w, dtype=torch.float64, device=dev).view(-1, 1, 1, 1)
        return {"f": torch.stack(g) + w}
    out = {"state": torch.stack(f if case["layout"] == "AB" else g)}
    if call == "march":
        del f
        out.update(X.diagnostics(g))
    elif call == "drag":
        out["force"] = X.drag(g)
    return out


def _exact_batch(case, seed, dev):
    e = ESIZE[case["storage"]]
    parts = []
    r = _rng(seed)
    for nx, ny, nu in _batch_members(case, _rng(1000 + case["lattices"])):
        rho, u = _fields(nx, ny, 1, 2, "shear", r, dev)
        X = _Exact(case, (1, ny, nx), nu, None, dev)
        g = X.equilibrium(rho, [u[0], u[1]])
        for s in range(case["steps"]):
            f = X.collide(g)
            g = X.stream(f)
        per = 16 // e
        pitch = (nx + per - 1) // per * per
        plane = (pitch * ny + 256 // e - 1) // (256 // e) * (256 // e)
        t = torch.zeros((9, plane), dtype=torch.float64, device=dev)
        t[:, :pitch * ny].view(9, ny, pitch)[..., :nx] = torch.stack(f)[:, 0]
        parts.append(t.view(-1))
    return {"state": torch.cat(parts)}
