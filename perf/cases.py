"""The work a user of the library has it do, as measurable cases.

A case names one call pattern of the public binding (``lbm.Simulation`` /
``lbm.AxiSimulation``) and its sizes. ``prepare`` builds the handle and loads a
seeded state into it (what a program restarting from a checkpoint does),
``run`` makes one pass, ``work`` states the bytes and operations the pass
cannot do without, and ``exact`` computes the same outputs in 64 bits from the
method's equations with plain torch.

Kinds of pass:

* ``step``      n time steps of one simulation, then the fields a user plots
                or feeds on: n, n p, and the raw Yee E and B;
* ``monitor``   n single steps with the fused FP64 diagnostics of each read
                on the host (a run that watches its own stability), then the
                same fields;
* ``window``    n steps with the box following the driver, then every output
                the library offers of a state: all 16 node fields, the FP64
                diagnostics, and the line cut with the bubble length;
* ``exchange``  the full state out of the library and back in (checkpoint and
                restart);
* ``scan``      n steps of many independent instances in one handle, then the
                fields of each;
* ``adjoint``   record n steps, read E, reverse sweep for the gradient of
                sum(seed E) with respect to the driver;
* ``axi``       n steps of the 2D-axisymmetric form, then its six fields.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2201_05473_gb300 import lbm
from paper_2201_05473_gb300 import workloads as W

STORAGE = {"f32": W.F32, "bf16": W.BF16, "f16": W.F16}
COLLISION = {"bgk": W.BGK, "regularized": W.REGULARIZED}
FIELDS = (lbm.FIELD_N | lbm.FIELD_PX | lbm.FIELD_PY | lbm.FIELD_PZ | lbm.FIELD_EX | lbm.FIELD_EY | lbm.FIELD_EZ
          | lbm.FIELD_BX | lbm.FIELD_BY | lbm.FIELD_BZ | lbm.RAW_YEE)
ALL_FIELDS = 0xFFFF

# D3Q19 in the library's order (include/pwfa_lbm.h), and D2Q9 as (z, r)
XI = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
      (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
      (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
WQ = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12
XI9 = [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (-1, -1), (1, -1), (-1, 1)]
W9 = [4.0 / 9.0] + [1.0 / 9.0] * 4 + [1.0 / 36.0] * 4


# ---------------------------------------------------------------- the cases
def _grid(nz, ny, nx):
    return {"nz": nz, "ny": ny, "nx": nx}


def listed():
    return [
        # the parity workload: a quick look at a small wake, where launches
        # and latency count (200 steps in the repository's configuration)
        {"name": "small", "kind": "step", **_grid(64, 32, 32), "dx": 0.2, "tau": 0.51, "alpha": 0.1,
         "sigma_r": 0.5, "sigma_z": 0.5, "collision": "bgk", "storage": "f32", "steps": 50},
        # an exploratory run on a grid cut to the plasma at hand: odd sizes
        # that no tile divides, an odd number of steps
        {"name": "ragged", "kind": "step", **_grid(203, 97, 131), "dx": 0.1, "tau": 0.53, "alpha": 0.5,
         "sigma_r": 0.4, "sigma_z": 0.5, "collision": "bgk", "storage": "f32", "steps": 21},
        # the production run (2000 steps of it make a result), FP32
        {"name": "production", "kind": "step", **_grid(512, 256, 256), "dx": 0.05, "tau": 0.53, "alpha": 1.0,
         "sigma_r": 0.3, "sigma_z": 0.5, "collision": "regularized", "storage": "f32", "steps": 20},
        # the production run in the reduced-precision form that meets 1e-3
        {"name": "production_f16", "kind": "step", **_grid(512, 256, 256), "dx": 0.05, "tau": 0.53,
         "alpha": 1.0, "sigma_r": 0.3, "sigma_z": 0.5, "collision": "regularized", "storage": "f16", "steps": 20},
        # the precision form: linear driver, BGK, BF16 storage
        {"name": "precision_bf16", "kind": "step", **_grid(256, 128, 128), "dx": 0.2, "tau": 0.51, "alpha": 0.1,
         "sigma_r": 0.5, "sigma_z": 0.5, "collision": "bgk", "storage": "bf16", "steps": 40},
        # a monitored run: every step's diagnostics come back to the host
        # (the end-to-end line of the benchmark)
        {"name": "monitor", "kind": "monitor", **_grid(256, 128, 128), "dx": 0.1, "tau": 0.53, "alpha": 0.5,
         "sigma_r": 0.4, "sigma_z": 0.5, "collision": "regularized", "storage": "f32", "steps": 10},
        # a long propagation in the moving window, observed after some steps
        {"name": "window", "kind": "window", **_grid(256, 128, 128), "dx": 0.1, "tau": 0.53, "alpha": 0.5,
         "sigma_r": 0.4, "sigma_z": 0.5, "collision": "regularized", "storage": "f32", "steps": 24},
        # checkpoint and restart
        {"name": "exchange", "kind": "exchange", **_grid(256, 128, 128), "dx": 0.2, "tau": 0.51, "alpha": 0.1,
         "sigma_r": 0.5, "sigma_z": 0.5, "collision": "bgk", "storage": "f32", "steps": 0},
        # a parameter scan over uneven grids (half of the repository's 64)
        {"name": "scan", "kind": "scan", "instances": 32, "draw_seed": 0, "small": False, "collision": "bgk",
         "storage": "f32", "steps": 10},
        # a scan of many instances too small to fill the GPU alone
        {"name": "scan_small", "kind": "scan", "instances": 256, "draw_seed": 0, "small": True,
         "collision": "bgk", "storage": "f32", "steps": 100},
        # the differentiable form: forward with checkpoints, then the sweep
        {"name": "adjoint", "kind": "adjoint", **_grid(256, 128, 128), "dx": 0.2, "tau": 0.51, "alpha": 0.5,
         "sigma_r": 0.5, "sigma_z": 0.5, "collision": "bgk", "storage": "f32", "steps": 40},
        # the paper's own geometry on the paper's grid
        {"name": "axisymmetric", "kind": "axi", "nz": 2400, "nr": 402, "dx": 0.25 / W.KP_INV_UM, "tau": 0.51,
         "alpha": 0.68, "sigma_r": 8.9 / W.KP_INV_UM, "sigma_z": 17.7 / W.KP_INV_UM, "steps": 100},
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "monitor", "window", "exchange", "scan", "scan", "adjoint",
                       "axi"])
    if kind == "axi":
        cells = math.exp(rng.uniform(math.log(64 * 34), math.log(2400 * 402)))
        aspect = math.exp(rng.uniform(math.log(1.5), math.log(7.0)))
        nr = max(10, int(round(math.sqrt(cells / aspect))))
        return {"kind": kind, "nz": max(16, int(cells / nr)), "nr": nr, "dx": rng.choice([0.2, 0.05, 0.01]),
                "tau": 0.51, "alpha": rng.uniform(0.1, 0.68), "sigma_r": rng.uniform(0.2, 0.5),
                "sigma_z": rng.uniform(0.3, 0.5), "steps": rng.randint(20, 100)}
    collision = rng.choice(["bgk", "regularized"])
    storage = rng.choice(["f32", "f32", "bf16", "f16"])
    if kind == "scan":
        small = rng.random() < 0.5
        return {"kind": kind, "instances": rng.randint(16, 256) if small else rng.randint(2, 24),
                "draw_seed": rng.randint(1, 10 ** 6), "small": small, "collision": collision, "storage": storage,
                "steps": rng.randint(8, 60) if small else rng.randint(2, 10)}
    top = {"step": 512 * 256 * 256, "monitor": 256 * 128 * 128, "window": 256 * 128 * 128,
           "exchange": 256 * 128 * 128, "adjoint": 128 * 96 * 96}[kind]
    nodes = math.exp(rng.uniform(math.log(64 * 32 * 32), math.log(top)))
    nx = max(8, int(round((nodes / 2.0) ** (1.0 / 3.0) * rng.uniform(0.7, 1.3))))
    ny = max(8, int(round((nodes / 2.0) ** (1.0 / 3.0) * rng.uniform(0.7, 1.3))))
    if rng.random() < 0.4:
        nx += (-nx) % 32
    nz = min(max(16, int(nodes / (nx * ny))), max(16, top // (nx * ny)))
    steps = {"step": rng.randint(1, 20), "monitor": rng.randint(1, 10), "window": rng.randint(6, 24),
             "exchange": 0, "adjoint": rng.randint(4, 30)}[kind]
    return {"kind": kind, "nz": nz, "ny": ny, "nx": nx, "dx": rng.choice([0.2, 0.1, 0.05]), "tau": 0.55,
            "alpha": rng.uniform(0.1, 1.0), "sigma_r": rng.uniform(0.3, 0.6), "sigma_z": rng.uniform(0.3, 0.6),
            "collision": collision, "storage": "f32" if kind == "adjoint" else storage, "steps": steps}


# ---------------------------------------------------------------- inputs
def _workload(case, seed):
    """The single-instance workload: the driver inside the box, its strength
    and sizes varied with the seed."""
    r = np.random.default_rng([seed, 11])
    v = r.uniform(0.9, 1.1, size=3)
    w = W.Workload(nx=case["nx"], ny=case["ny"], nz=case["nz"], dx=case["dx"], tau=case["tau"],
                   alpha=case["alpha"] * v[0], sigma_r=case["sigma_r"] * v[1], sigma_z=case["sigma_z"] * v[2],
                   z0=0.6 * case["nz"] * case["dx"], steps=case["steps"], collision=COLLISION[case["collision"]],
                   storage=STORAGE[case["storage"]])
    if case["kind"] == "window":
        # the driver reaches window_z during the first cell it crosses
        w = w.replace(moving_window=1, window_z=w.z0 + 0.3 * case["dx"])
    return w


def _scan_workloads(case, seed):
    ws = (W.small_scan if case["small"] else W.batched_scan)(case["instances"], seed=case["draw_seed"],
                                                             steps=case["steps"])
    r = np.random.default_rng([seed, 12])
    return [w.replace(alpha=w.alpha * float(r.uniform(0.8, 1.2)), z0=0.6 * w.nz * w.dx,
                      collision=COLLISION[case["collision"]], storage=STORAGE[case["storage"]]) for w in ws]


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _state(w, seed, tag=0):
    """A plasma carrying waves: densities, momenta and fields as sums of a few
    smooth modes, populations at the equilibrium of those moments plus a
    small non-equilibrium part. float32 (f [4][19][z][y][x], E, B [3][z][y][x])."""
    dev = _device()
    shp = (w.nz, w.ny, w.nx)
    r = np.random.default_rng([seed, 13, tag])
    gen = torch.Generator(device=dev).manual_seed(int(r.integers(1 << 40)))

    def smooth(amp):
        out = torch.zeros(shp, dtype=torch.float32, device=dev)
        for _ in range(3):
            ax = []
            for n in shp:
                k, ph = r.uniform(0.5, 4.0), r.uniform(0.0, 2.0 * math.pi)
                ax.append(torch.from_numpy(np.cos(2.0 * math.pi * k * np.arange(n) / n + ph).astype(np.float32))
                          .to(dev))
            out += (amp / 3.0) * (ax[0][:, None, None] * ax[1][None, :, None] * ax[2][None, None, :])
        return out

    A = [1.0 + smooth(0.1)] + [smooth(0.05) for _ in range(3)]
    p = [A[k] / A[0] for k in (1, 2, 3)]
    ig = torch.rsqrt(1.0 + p[0] ** 2 + p[1] ** 2 + p[2] ** 2)
    lat = W.DT_OVER_DX
    u = [c * ig * lat for c in p]
    base = 1.0 - 1.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
    f = torch.empty((4, 19) + shp, dtype=torch.float32, device=dev)
    for q, (cx, cy, cz) in enumerate(XI):
        xu = cx * u[0] + cy * u[1] + cz * u[2]
        phi = WQ[q] * (base + 3.0 * xu + 4.5 * xu * xu)
        for k in range(4):
            f[k, q] = A[k] * phi + 1e-4 * WQ[q] * torch.randn(shp, generator=gen, device=dev)
    E = torch.stack([smooth(0.05) for _ in range(3)])
    B = torch.stack([smooth(0.02) for _ in range(3)])
    return f, E, B


def _seed_E(case, seed):
    """dL/dE of the gradient cases: a smooth weight around the driver."""
    w = _workload(case, seed)
    r = np.random.default_rng([seed, 14])
    ax = []
    for n, c, s in ((w.nz, 0.6 + 0.05 * r.uniform(-1, 1), 0.15), (w.ny, 0.5, 0.2), (w.nx, 0.5, 0.2)):
        t = np.arange(n) / n
        ax.append(np.exp(-0.5 * ((t - c) / s) ** 2))
    g = ax[0][:, None, None] * ax[1][None, :, None] * ax[2][None, None, :]
    amp = r.uniform(0.5, 1.0, size=3)
    return torch.from_numpy((amp[:, None, None, None] * g[None]).astype(np.float32)).to(_device())


def _axi_workload(case, seed):
    r = np.random.default_rng([seed, 15])
    v = r.uniform(0.9, 1.1, size=3)
    return W.AxiWorkload(nz=case["nz"], nr=case["nr"], dx=case["dx"], tau=case["tau"], alpha=case["alpha"] * v[0],
                         sigma_r=case["sigma_r"] * v[1], sigma_z=case["sigma_z"] * v[2],
                         z0=0.6 * case["nz"] * case["dx"], steps=case["steps"])


def _axi_source(w, seed):
    """Streaming source [3][9][nz][nr] of a plasma with smooth density and
    momentum waves (row 0 the mirror image of row 1)."""
    r = np.random.default_rng([seed, 16])
    z, j = np.arange(w.nz) / w.nz, (np.arange(w.nr) - 0.5) / w.nr

    def smooth(amp, odd=False):
        out = np.zeros((w.nz, w.nr))
        for _ in range(3):
            kz, ph, kr = r.uniform(0.5, 4.0), r.uniform(0.0, 2.0 * math.pi), r.uniform(0.5, 2.0)
            rad = np.sin(math.pi * kr * j) if odd else np.cos(math.pi * kr * j)
            out += (amp / 3.0) * np.cos(2.0 * math.pi * kz * z + ph)[:, None] * rad[None, :]
        return out

    A = [1.0 + smooth(0.1), smooth(0.03), smooth(0.03, odd=True)]
    S = np.empty((3, 9, w.nz, w.nr), dtype=np.float32)
    for q in range(9):
        for k in range(3):
            S[k, q] = W9[q] * A[k]
    refl = [0, 1, 2, 4, 3, 7, 8, 5, 6]
    for q in range(9):
        for k in range(3):
            S[k, refl[q], :, 0] = (-1.0 if k == 2 else 1.0) * S[k, q, :, 1]
    return torch.from_numpy(S).to(_device())


def prepare(case, seed):
    kind = case["kind"]
    if kind == "axi":
        w = _axi_workload(case, seed)
        sim = lbm.AxiSimulation(w)
        sim.set_source(_axi_source(w, seed))
        return {"case": case, "sim": sim}
    if kind == "scan":
        ws = _scan_workloads(case, seed)
        sim = lbm.Simulation(ws)
        for i, w in enumerate(ws):
            sim.set_state(*_state(w, seed, i), instance=i)
        return {"case": case, "sim": sim}
    sim = lbm.Simulation(_workload(case, seed))
    st = {"case": case, "sim": sim}
    if kind == "adjoint":
        st["seed_E"] = _seed_E(case, seed)  # the recording starts from rest
    else:
        sim.set_state(*_state(sim.works[0], seed))
    return st


# ---------------------------------------------------------------- one pass
def run(state):
    case, sim = state["case"], state["sim"]
    kind, steps = case["kind"], case["steps"]
    if kind == "step":
        sim.step(steps)
        return sim.fields(FIELDS)
    if kind == "monitor":
        diags = np.empty((steps, 8))
        for k in range(steps):
            sim.step_diag(1, out=diags[k:k + 1])
        return {"diag": diags, "fields": sim.fields(FIELDS)}
    if kind == "window":
        sim.step(steps)
        out = sim.fields(ALL_FIELDS)
        n, ez, length = sim.linecut()
        return {"fields": out, "diag": sim.diag(), "line_n": n, "line_ez": ez, "bubble_length": length}
    if kind == "exchange":
        f, E, B = sim.get_state()
        sim.set_state(f, E, B)
        return [f, E, B]
    if kind == "scan":
        sim.step(steps)
        if not case["small"]:
            return [sim.fields(FIELDS, instance=i) for i in range(case["instances"])]
        # equal grids: one array over the instances
        out = torch.empty((case["instances"], 10) + sim.shape(0), dtype=torch.float32, device=_device())
        for i in range(case["instances"]):
            sim.fields(FIELDS, instance=i, out=out[i])
        return out
    if kind == "adjoint":
        sim.record(steps)
        E = sim.fields(lbm.FIELD_EX | lbm.FIELD_EY | lbm.FIELD_EZ | lbm.RAW_YEE)
        return {"E": E, "grad": sim.adjoint_step(state["seed_E"])}
    sim.step(steps)
    return sim.fields()


# ---------------------------------------------------------------- floors
# operations of one node-step: moments 76, shared equilibrium factors ~110,
# collision and source ~6 per population (BGK) or ~5 (regularized), node
# fields and force ~60, Yee updates ~45, velocity and current ~40
_FLOPS = {"bgk": 790.0, "regularized": 830.0}


def work(case):
    kind, steps = case["kind"], case["steps"]
    if kind == "axi":
        N = case["nz"] * case["nr"]
        # source, E_z, E_r, B_theta in and out, six fields out
        return {"bytes": float(N * (2 * (27 + 3) * 4 + 6 * 4)), "flops": float(N * steps * 330)}
    ws = _scan_workloads(case, 0) if kind == "scan" else [_workload(case, 0)]
    N = sum(w.nodes for w in ws)
    pop = 76 * (4 if case["storage"] == "f32" else 2)
    fl = _FLOPS[case["collision"]]
    state = pop + 24  # the populations, E and B of one node
    if kind == "exchange":
        # stored state and FP32 arrays, each read once and written once
        return {"bytes": float(N * 2 * (state + 328)), "flops": float(N * 76)}
    if kind == "adjoint":
        # the seed read, E written; the run itself starts from rest and ends
        # with a gradient: the final state and the adjoint of the initial
        # one written once. A reversed step costs about two forward ones.
        return {"bytes": float(N * (12 + 12 + state + 304)), "flops": float(N * steps * 3 * fl)}
    out = {"step": 40, "monitor": 40, "scan": 40, "window": 64}[kind]
    return {"bytes": float(N * (2 * state + out)), "flops": float(N * steps * fl)}


# ---------------------------------------------------------------- 64 bits
class _Box:
    """The 3D scheme on one open box (or a batch of equal boxes, leading
    axis) in float64. Arrays end in [z][y][x]; S is the streaming source."""

    def __init__(self, shape, dx, tau, collision, alpha, sigma_r, sigma_z, z0, window=None, batch=()):
        self.nz, self.ny, self.nx = shape
        self.batch, self.dx, self.dt, self.tau, self.collision = batch, dx, W.DT_OVER_DX * dx, tau, collision
        self.alpha, self.sr, self.sz, self.z0, self.window = alpha, sigma_r, sigma_z, z0, window
        self.n = 0
        dev = _device()
        idx = [torch.arange(m, dtype=torch.float64, device=dev) for m in shape]
        self.z = (idx[0] + 0.5)[:, None, None] * dx
        y = (idx[1] - 0.5 * (self.ny - 1))[None, :, None] * dx
        x = (idx[2] - 0.5 * (self.nx - 1))[None, None, :] * dx
        self.r2 = x * x + y * y
        full = batch + tuple(shape)
        z64 = lambda *lead: torch.zeros(lead + full, dtype=torch.float64, device=dev)
        self.S, self.E, self.B, self.J = z64(4, 19), z64(3), z64(3), z64(3)
        for q in range(19):
            self.S[0, q] = WQ[q]

        def mask(inx, iny, inz):
            # True where a Yee component is free: the index ranges of the
            # axes along which it must lie off both walls (1..n-2) or only
            # below the far one (0..n-2)
            m = torch.ones(tuple(shape), dtype=torch.bool, device=dev)
            for ax, off in ((2, inx), (1, iny), (0, inz)):
                sl = [slice(None)] * 3
                sl[ax] = -1
                m[tuple(sl)] = False
                if off:
                    sl[ax] = 0
                    m[tuple(sl)] = False
            return m
        self.mE = [mask(0, 1, 1), mask(1, 0, 1), mask(1, 1, 0)]
        self.mB = [mask(1, 0, 0), mask(0, 1, 0), mask(0, 0, 1)]

    def walls(self):
        for c in range(3):
            self.E[c] = torch.where(self.mE[c], self.E[c], 0.0)
            self.B[c] = torch.where(self.mB[c], self.B[c], 0.0)

    def load(self, f, E, B):
        """Import a pre-collision state: S_i(y) = f_i(y + xi_i), indices past
        the box clamped into it."""
        for q, (cx, cy, cz) in enumerate(XI):
            g = f[:, q].double()
            for ax, c in ((-1, cx), (-2, cy), (-3, cz)):
                if c:
                    n = g.shape[ax]
                    i = (torch.arange(n, device=g.device) + c).clamp(0, n - 1)
                    g = g.index_select(g.dim() + ax, i)
            self.S[:, q] = g
        self.E, self.B = E.double().clone(), B.double().clone()
        self.walls()

    @staticmethod
    def clamp_nodes(a):
        """Boundary nodes take their clamped interior node's values."""
        for ax in (-1, -2, -3):
            n = a.shape[ax]
            i = torch.arange(n, device=a.device).clamp(1, n - 2)
            a = a.index_select(a.dim() + ax, i)
        return a

    def pulled(self, l, q):
        """f_{l,q} at interior nodes, clamped to the boundary ones."""
        cx, cy, cz = XI[q]
        return self.clamp_nodes(torch.roll(self.S[l, q], shifts=(cz, cy, cx), dims=(-3, -2, -1)))

    def moments(self):
        return [sum(self.pulled(l, q) for q in range(19)) for l in range(4)]

    @staticmethod
    def velocity(A):
        n = torch.clamp(A[0], min=1e-6)
        p = [A[k] / n for k in (1, 2, 3)]
        ig = 1.0 / torch.sqrt(1.0 + p[0] ** 2 + p[1] ** 2 + p[2] ** 2)
        return n, [c * ig for c in p]

    @staticmethod
    def shift(a, ax, d):
        """a at index + d along ax (x, y, z = -1, -2, -3), zero outside."""
        out = torch.zeros_like(a)
        n = a.shape[ax]
        if d > 0:
            out.narrow(ax, 0, n - d).copy_(a.narrow(ax, d, n - d))
        else:
            out.narrow(ax, -d, n + d).copy_(a.narrow(ax, 0, n + d))
        return out

    def planes(self, n):
        if self.window is None:
            return 0
        return max(0, math.floor((self.z0 + n * self.dt - self.window) / self.dx))

    def move(self):
        """The box moves one plane along +z: source and fields one plane
        down, plasma at rest and no field on the top plane."""
        top = torch.zeros_like(self.S[..., :1, :, :])
        for q in range(19):
            top[0, q] = WQ[q]
        self.S = torch.cat([self.S[..., 1:, :, :], top], dim=-3)
        self.E, self.B = self.shift(self.E, -3, 1), self.shift(self.B, -3, 1)
        self.walls()

    def node_E(self):
        return [0.5 * (self.shift(self.E[c], -1 - c, -1) + self.E[c]) for c in range(3)]

    def node_B(self, B):
        out = []
        for c in range(3):
            a, b = [ax for ax in (-1, -2, -3) if ax != -1 - c]
            t = B[c] + self.shift(B[c], a, -1)
            out.append(0.25 * (t + self.shift(t, b, -1)))
        return out

    def step(self):
        c, dt = self.dt / self.dx, self.dt
        w1 = self.planes(self.n + 1)
        if w1 > self.planes(self.n):
            self.move()
        E, B = self.E, self.B
        d = lambda a, ax: self.shift(a, ax, 1) - a
        X, Y, Z = -1, -2, -3
        curl = [d(E[2], Y) - d(E[1], Z), d(E[0], Z) - d(E[2], X), d(E[1], X) - d(E[0], Y)]
        Bn = torch.stack([torch.where(self.mB[k], B[k] - c * curl[k], 0.0) for k in range(3)])
        # fluid
        f = [[self.pulled(l, q) for q in range(19)] for l in range(4)]
        A = [sum(f[l]) for l in range(4)]
        n, beta = self.velocity(A)
        e, b = self.node_E(), self.node_B(0.5 * (B + Bn))
        F = [-A[0] * (e[0] + beta[1] * b[2] - beta[2] * b[1]),
             -A[0] * (e[1] + beta[2] * b[0] - beta[0] * b[2]),
             -A[0] * (e[2] + beta[0] * b[1] - beta[1] * b[0])]
        u = [v * c for v in beta]
        base = 1.0 - 1.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        phi = []
        for q, (cx, cy, cz) in enumerate(XI):
            xu = cx * u[0] + cy * u[1] + cz * u[2]
            phi.append(WQ[q] * (base + 3.0 * xu + 4.5 * xu * xu))
        inner = torch.zeros((self.nz, self.ny, self.nx), dtype=torch.bool, device=self.r2.device)
        inner[1:-1, 1:-1, 1:-1] = True
        S = torch.empty_like(self.S)
        for l in range(4):
            # a boundary node holds the equilibrium of its clamped node
            fl = [torch.where(inner, f[l][q], A[l] * phi[q]) for q in range(19)]
            f[l] = None
            src = F[l - 1] * dt if l else 0.0
            if self.collision == W.REGULARIZED:
                k3 = 3.0 * (1.0 - 1.0 / self.tau)
                P = [k3 * (sum(XI[q][k] * fl[q] for q in range(1, 19) if XI[q][k]) - A[l] * u[k]) for k in range(3)]
            for q in range(19):
                if self.collision == W.BGK:
                    v = fl[q] + (A[l] * phi[q] - fl[q]) / self.tau + WQ[q] * src
                else:
                    v = A[l] * phi[q] + WQ[q] * (src + sum(XI[q][k] * P[k] for k in range(3) if XI[q][k]))
                S[l, q] = v
        self.S = S
        ps = [(A[k + 1] + F[k] * dt) / n for k in range(3)]
        ng = -A[0] / torch.sqrt(1.0 + ps[0] ** 2 + ps[1] ** 2 + ps[2] ** 2)
        J = torch.stack([ng * v for v in ps])
        # Ampere with the driver at t_{n+1}
        zc = self.z0 + (self.n + 1) * dt - w1 * self.dx
        nb = self.alpha * torch.exp(-self.r2 / (2.0 * self.sr ** 2) - (self.z - zc) ** 2 / (2.0 * self.sz ** 2))
        g = lambda a, ax: a - self.shift(a, ax, -1)
        cb = [g(Bn[2], Y) - g(Bn[1], Z), g(Bn[0], Z) - g(Bn[2], X), g(Bn[1], X) - g(Bn[0], Y)]
        En = []
        for k in range(3):
            je = 0.5 * (J[k] + self.shift(J[k], -1 - k, 1))
            if k == 2:
                je = je - nb
            En.append(torch.where(self.mE[k], E[k] + c * cb[k] - dt * je, E[k]))
        self.E, self.B, self.J = torch.stack(En), Bn, J
        self.n += 1

    def diag(self):
        """The eight diagnostics of the current state."""
        A = self.moments()
        _, beta = self.velocity(A)
        en = 0.5 * ((self.E ** 2).sum() + (self.B ** 2).sum()) * self.dx ** 3
        v = [A[0].sum(), A[1].sum(), A[2].sum(), A[3].sum(), en, A[0].min(),
             torch.sqrt(beta[0] ** 2 + beta[1] ** 2 + beta[2] ** 2).max()]
        return np.array([float(t) for t in v] + [0.0])

    def fields(self):
        """The FIELDS outputs, in the mask's bit order."""
        A = self.moments()
        return torch.stack([A[0], *self.E, *self.B, *A[1:]])


def _exact_box(w):
    return _Box((w.nz, w.ny, w.nx), w.dx, w.tau, w.collision, w.alpha, w.sigma_r, w.sigma_z, w.z0,
                window=w.window_z if w.moving_window else None)


def _exact_axi(case, seed):
    w = _axi_workload(case, seed)
    S = _axi_source(w, seed).double()
    nz, nr, dx, dt, tau = w.nz, w.nr, w.dx, w.dt, w.tau
    c, dev = dt / dx, S.device
    D = (tau - 0.5) / 3.0 * dx * dx / dt
    zero = lambda: torch.zeros((nz, nr), dtype=torch.float64, device=dev)
    Ez, Er, Bt, Jz, Jr = zero(), zero(), zero(), zero(), zero()
    j = torch.arange(nr, dtype=torch.float64, device=dev)[None, :]
    r = (j - 0.5) * dx
    zed = (torch.arange(nz, dtype=torch.float64, device=dev) + 0.5)[:, None] * dx
    kc = torch.arange(nz, device=dev).clamp(1, nz - 2)
    jc = torch.arange(nr, device=dev).clamp(1, nr - 2)
    bnd = torch.zeros((nz, nr), dtype=torch.bool, device=dev)
    bnd[0], bnd[-1], bnd[:, -1] = True, True, True
    refl = [0, 1, 2, 4, 3, 7, 8, 5, 6]

    def shift(a, ax, d):
        return _Box.shift(a, ax, d)

    def pulled():
        return [[torch.roll(S[l, q], shifts=XI9[q], dims=(0, 1)).index_select(0, kc).index_select(1, jc)
                 for q in range(9)] for l in range(3)]

    def velocity(A):
        n = torch.clamp(A[0], min=1e-6)
        pz, pr = A[1] / n, A[2] / n
        ig = 1.0 / torch.sqrt(1.0 + pz * pz + pr * pr)
        return n, pz * ig, pr * ig

    for n in range(w.steps):
        f = pulled()
        A = [sum(f[l]) for l in range(3)]
        A[2] = torch.cat([-A[2][:, :1], A[2][:, 1:]], dim=1)
        act = torch.zeros((nz, nr), dtype=torch.bool, device=dev)
        act[:nz - 1, 1:nr - 1] = True
        Bn = torch.where(act, Bt - c * ((shift(Er, -2, 1) - Er) - (shift(Ez, -1, 1) - Ez)), 0.0)
        _, bz, br = velocity(A)
        uz, ur = bz * c, br * c
        phi = []
        for q, (cz, cr) in enumerate(XI9):
            xu = cz * uz + cr * ur
            phi.append(W9[q] * (1.0 + 3.0 * xu + 4.5 * xu * xu - 1.5 * (uz * uz + ur * ur)))
        ez = 0.5 * (shift(Ez, -2, -1) + Ez)
        er = 0.5 * (shift(Er, -1, -1) + Er)
        t = Bt + Bn
        t = t + shift(t, -2, -1)
        bt = 0.125 * (t + shift(t, -1, -1))
        src = [torch.zeros_like(bz), -A[0] * (ez + br * bt), -A[0] * (er - bz * bt)]
        for l in range(3):
            cyl = (0.5 * D / dx * (shift(A[l], -1, 1) - shift(A[l], -1, -1)) - A[l] * br) / r
            src[l] = src[l] + torch.where(bnd, 0.0, cyl)
        new = torch.empty_like(S)
        for l in range(3):
            for q in range(9):
                fl = torch.where(bnd, A[l] * phi[q], f[l][q])
                new[l, q] = fl + (A[l] * phi[q] - fl) / tau + W9[q] * src[l] * dt
        sg = [1.0, 1.0, -1.0]
        for l in range(3):
            for q in range(9):
                new[l, refl[q], :, 0] = sg[l] * new[l, q, :, 1]
        S = new
        st = [A[l] + src[l] * dt for l in range(3)]
        _, cz, cr = velocity(st)
        Jz, Jr = -st[0] * cz, -st[0] * cr
        Jz[:, 0], Jr[:, 0] = Jz[:, 1], -Jr[:, 1]
        zc = w.z0 + (n + 1) * dt
        nb = w.alpha * torch.exp(-r * r / (2 * w.sigma_r ** 2) - (zed - zc) ** 2 / (2 * w.sigma_z ** 2))
        mr = torch.zeros_like(act)
        mr[1:nz - 1, 1:nr - 1] = True
        Ern = torch.where(mr, Er - c * (Bn - shift(Bn, -2, -1)) - dt * 0.5 * (Jr + shift(Jr, -1, 1)), Er)
        curl = (j * Bn - (j - 1.0) * shift(Bn, -1, -1)) / (j - 0.5)
        Ez = torch.where(act, Ez + c * curl - dt * (0.5 * (Jz + shift(Jz, -2, 1)) - nb), Ez)
        Er, Bt = Ern, Bn
    A = [sum(fl) for fl in pulled()]
    A[2] = torch.cat([-A[2][:, :1], A[2][:, 1:]], dim=1)
    _, bz, br = velocity(A)
    return torch.stack([A[0], bz, br, Ez, Er, Bt])


def _exact_adjoint(case, seed):
    """dL/d(alpha, sigma_r, sigma_z) of L = sum(seed E), one forward-mode
    derivative each."""
    import torch.autograd.forward_ad as fwd
    w = _workload(case, seed)
    sE = _seed_E(case, seed).double()
    dev = sE.device
    grad, E = np.zeros(3), None
    for k in range(3):
        with fwd.dual_level(), torch.no_grad():
            p = [torch.tensor(v, dtype=torch.float64, device=dev) for v in (w.alpha, w.sigma_r, w.sigma_z)]
            p[k] = fwd.make_dual(p[k], torch.ones_like(p[k]))
            box = _Box((w.nz, w.ny, w.nx), w.dx, w.tau, w.collision, p[0], p[1], p[2], w.z0)
            for _ in range(case["steps"]):
                box.step()
            t = fwd.unpack_dual(box.E)
            E = t.primal.detach().clone()
            grad[k] = float((sE * t.tangent).sum())
    return {"E": E, "grad": grad}


def exact(case, seed):
    kind, steps = case["kind"], case["steps"]
    with torch.no_grad():
        if kind == "axi":
            return _exact_axi(case, seed)
        if kind == "adjoint":
            return _exact_adjoint(case, seed)
        if kind == "scan":
            ws = _scan_workloads(case, seed)
            if case["small"]:
                # equal grids: the boxes as one batch
                dev = _device()
                col = lambda k: torch.tensor([getattr(w, k) for w in ws], dtype=torch.float64,
                                             device=dev)[:, None, None, None]
                w0 = ws[0]
                box = _Box((w0.nz, w0.ny, w0.nx), w0.dx, w0.tau, w0.collision, col("alpha"), col("sigma_r"),
                           col("sigma_z"), w0.z0, batch=(len(ws),))
                st = [_state(w, seed, i) for i, w in enumerate(ws)]
                box.load(*[torch.stack([s[k] for s in st], dim=(2 if k == 0 else 1)) for k in range(3)])
                for _ in range(steps):
                    box.step()
                return box.fields().transpose(0, 1).contiguous()
            outs = []
            for i, w in enumerate(ws):
                box = _exact_box(w)
                box.load(*_state(w, seed, i))
                for _ in range(steps):
                    box.step()
                outs.append(box.fields())
            return outs
        w = _workload(case, seed)
        box = _exact_box(w)
        box.load(*_state(w, seed))
        if kind == "exchange":
            A = box.moments()
            _, beta = box.velocity(A)
            u = [v * (box.dt / box.dx) for v in beta]
            base = 1.0 - 1.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
            inner = torch.zeros_like(A[0], dtype=torch.bool)
            inner[1:-1, 1:-1, 1:-1] = True
            f = torch.empty((4, 19) + tuple(A[0].shape), dtype=torch.float64, device=A[0].device)
            for q, (cx, cy, cz) in enumerate(XI):
                xu = cx * u[0] + cy * u[1] + cz * u[2]
                phi = WQ[q] * (base + 3.0 * xu + 4.5 * xu * xu)
                for l in range(4):
                    f[l, q] = torch.where(inner, box.pulled(l, q), A[l] * phi)
            return [f, box.E, box.B]
        if kind == "monitor":
            diags = np.empty((steps, 8))
            for k in range(steps):
                diags[k] = box.diag()
                box.step()
            return {"diag": diags, "fields": box.fields()}
        for _ in range(steps):
            box.step()
        if kind == "step":
            return box.fields()
        # window: every node field, the diagnostics, the axis line
        A = box.moments()
        _, beta = box.velocity(A)
        e, b = box.node_E(), box.node_B(box.B)
        out = torch.stack([A[0], *beta, *e, *b, *box.J, A[1], A[2], A[3]])

        def on_axis(a):
            ys, xs = 0.5 * (w.ny - 1), 0.5 * (w.nx - 1)
            y0, x0 = int(ys), int(xs)
            fy, fx = ys - y0, xs - x0
            y1, x1 = min(y0 + 1, w.ny - 1), min(x0 + 1, w.nx - 1)
            t = ((1 - fy) * ((1 - fx) * a[:, y0, x0] + fx * a[:, y0, x1])
                 + fy * ((1 - fx) * a[:, y1, x0] + fx * a[:, y1, x1]))
            return t.cpu().numpy()
        line = on_axis(A[0])
        return {"fields": out, "diag": box.diag(), "line_n": line, "line_ez": on_axis(e[2]),
                "bubble_length": None}
