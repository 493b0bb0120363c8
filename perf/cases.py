"""Workloads of the phase-field lattice Boltzmann library, as its users run them.

Each case is one unit of a user's work through the public API
(``paper_2512_01032_gb300.pflb``): advance a prepared lattice (or a batch of
them) by some steps and read back the fields that the user looks at.  Lattices keep their state between passes, as a running
simulation does, so a further pass continues where the last one ended.

``exact`` is the same method (arXiv 2512.01032, Eqs. 1-15) written as plain
64-bit torch operations over whole arrays.

Fields are returned in the precision that they were computed in: FP64 for
FP64 lattices, FP32 for FP32 lattices, BF16 for lattices whose populations
are stored in 16 bits.  Velocities are left out of the FP32 and 16-bit cases:
in these start-up flows they are 1e-4 and below, so that their relative
rounding error is set by the light phase's division by rho = 1e-3.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2512_01032_gb300 import pflb

# ------------------------------------------------------------------- cases


def listed():
    return [
        # The paper's static droplet check as a plain FP64 run: the smallest
        # lattice, all fields read back.
        dict(name="drop32_fp64", kind="drop", nx=32, ny=32, nz=32, R=8.0, storage="fp64",
             steps=40, diag=False),
        # A small FP32 droplet watched at every step: one step and one
        # diagnostics read per call (latency of the smallest calls).
        dict(name="monitor32_fp32", kind="monitor", nx=32, ny=32, nz=32, R=8.0, storage="fp32",
             steps=30),
        # Contact-angle slug between plates: a thin lattice, many short steps.
        dict(name="slug_fp32", kind="slug", nx=192, H=32, nz=4, theta=60.0, storage="fp32",
             steps=20),
        # Drop on a curved wall at 128^3, diagnostics in every step: the
        # headline workload of the benchmark.
        dict(name="sessile128_fp32", kind="sessile", n=128, theta=60.0, storage="fp32", steps=40,
             diag=True),
        # The same at half the resolution, plain steps.
        dict(name="sessile64_fp32", kind="sessile", n=64, theta=90.0, storage="fp32", steps=60,
             diag=False),
        # The same at 128^3 with populations stored in BF16.
        dict(name="sessile128_bf16", kind="sessile", n=128, theta=60.0, storage="bf16", steps=60,
             diag=False),
        # Capillary filling of a two-plate slit, FP16 storage.
        dict(name="slit_fp16", kind="slit", nx=1024, ny=64, nz=4, reservoir=128, theta=45.0,
             storage="fp16", steps=100),
        # Slug pushed through a constricted duct by a pressure difference
        # across open x boundaries.
        dict(name="duct_open_fp32", kind="duct", w=48, ratio=0.5, theta=120.0, storage="fp32",
             open=True, steps=25),
        # Droplet carried along a square channel of odd size by a body force.
        dict(name="channel_odd_fp32", kind="channel", nx=251, ny=67, R=24.0, theta=100.0, u=5e-4,
             storage="fp32", steps=40),
        # Eight uneven constricted ducts advanced together, BF16 storage.
        dict(name="batch_ducts_bf16", kind="batch", what="duct",
             sizes="48 52 58 63 71 80 88 96", storage="bf16", steps=33),
        # Ten uneven droplet-in-channel lattices of any length, FP32.
        dict(name="batch_channels_fp32", kind="batch", what="channel",
             sizes="96x32 133x41 180x48 202x57 231x64 257x45 284x38 312x52 350x33 384x36",
             storage="fp32", steps=33),
        # A large closed box: a drop in gas, the size at which memory traffic
        # is all that counts.
        dict(name="box256_fp32", kind="drop", nx=256, ny=192, nz=160, R=48.0, storage="fp32",
             steps=24, diag=False),
    ]


def _between(rng, lo, hi):
    """An integer in [lo, hi], spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["drop", "drop", "monitor", "slug", "sessile", "sessile", "slit", "duct",
                       "duct", "channel", "channel", "batch"])
    storage = rng.choice(["fp32", "fp32", "fp32", "bf16", "fp16"])
    theta = float(rng.randint(60, 130))
    if kind in ("drop", "monitor"):
        if kind == "drop" and rng.random() < 0.2:
            storage = "fp64"
        hi = 48 if storage == "fp64" or kind == "monitor" else 192
        nx, ny, nz = (_between(rng, 24, hi) for _ in range(3))
        c = dict(kind=kind, nx=nx, ny=ny, nz=nz, R=0.25 * min(nx, ny, nz) + 1.0, storage=storage,
                 steps=24 if hi > 48 else 30)
        return c if kind == "monitor" else dict(c, diag=rng.random() < 0.4)
    if kind == "slug":
        return dict(kind="slug", nx=_between(rng, 128, 512), H=_between(rng, 24, 64),
                    nz=rng.randint(3, 8), theta=theta, storage=storage, steps=20)
    if kind == "sessile":
        return dict(kind="sessile", n=_between(rng, 48, 144), theta=theta, storage=storage,
                    steps=32, diag=rng.random() < 0.5)
    if kind == "slit":
        return dict(kind="slit", nx=_between(rng, 384, 1536), ny=_between(rng, 24, 96),
                    nz=rng.randint(3, 8), reservoir=128, theta=float(rng.randint(30, 60)),
                    storage=rng.choice(["bf16", "fp16"]), steps=60)
    if kind == "duct":
        return dict(kind="duct", w=_between(rng, 36, 80), ratio=round(rng.uniform(0.4, 0.7), 2),
                    theta=float(rng.randint(90, 140)), storage=storage,
                    open=rng.random() < 0.6, steps=24)
    if kind == "channel":
        ny = _between(rng, 32, 96)
        return dict(kind="channel", nx=_between(rng, 96, 384), ny=ny,
                    R=round(rng.uniform(0.3, 0.42) * ny, 2), theta=theta,
                    u=round(rng.uniform(1e-4, 1e-3), 6), storage=storage, steps=32)
    what = rng.choice(["duct", "channel"])
    if what == "duct":
        sizes = " ".join(str(rng.randint(40, 88)) for _ in range(rng.randint(2, 6)))
    else:
        sizes = " ".join("%dx%d" % (rng.randint(96, 384), rng.randint(32, 64))
                         for _ in range(rng.randint(3, 10)))
    return dict(kind="batch", what=what, sizes=sizes, storage=storage, steps=25)


# -------------------------------------------------- geometry, inputs, plans

PLAIN = dict(F_mode=0, mobility_corr=1, free_slip=0, blend=0.0)
WETTED = dict(F_mode=1, mobility_corr=1, free_slip=1, blend=0.95)
DROP = dict(sigma=0.01, W=4.0, M=0.02, rho_H=1.0, rho_L=1e-3, nu_H=0.1, nu_L=0.1)
CAPILLARY = dict(sigma=0.01, W=4.0, M=0.1666, rho_H=1.0, rho_L=1e-3, nu_H=1.0 / 60.0,
                 nu_L=1.0 / 3.0)


def _flat_normals(shape, planes):
    """Unit normals of axis-aligned walls: planes = [(axis, index, sign)],
    the fluid layer at that index taking that normal."""
    n = np.zeros(shape + (3,))
    for axis, index, sign in planes:  # axis 0 = x, 1 = y, 2 = z
        at = [slice(None)] * 3
        at[2 - axis] = index
        n[tuple(at)] = 0.0
        n[tuple(at) + (axis,)] = sign
    return n


def _setup(c, seed):
    """One lattice of a case: sizes, mask, normals, angles, parameters,
    initial state and boundaries, for this seed."""
    rng = np.random.Generator(np.random.PCG64(seed))
    jit = lambda s=1.0: float(rng.uniform(-s, s))  # noqa: E731
    kind = c["kind"]
    s = dict(storage=c["storage"], normals=None, theta=None, bounds=None)
    if kind in ("drop", "monitor"):
        # A drop in its own vapour, periodic box; centre off the lattice
        # sites, radius within 5 %.
        nx, ny, nz = c["nx"], c["ny"], c["nz"]
        s.update(dims=(nx, ny, nz), solid=None, params=dict(DROP, **PLAIN),
                 init=dict(shape=0, center=((nx - 1) / 2 + 0.3 * jit(), (ny - 1) / 2 + 0.3 * jit(),
                                            (nz - 1) / 2 + 0.3 * jit()),
                           R=c["R"] * (1 + 0.05 * jit())))
        return s
    if kind == "sessile":
        # A drop tangent to a solid ball on the floor of a closed box.
        n, k = c["n"], c["n"] / 128.0
        m = (n - 1) / 2.0
        z, y, x = np.meshgrid(*([np.arange(n, dtype=float)] * 3), indexing="ij", sparse=True)
        r = np.sqrt((x - m) ** 2 + (y - m) ** 2 + z ** 2)
        solid = r < 30.0 * k
        solid[0] = True
        solid[n - 1] = True
        near = r - 30.0 * k < np.minimum(z - 0.5, n - 1.5 - z)  # nearest wall: the ball
        nrm = np.zeros((n, n, n, 3))
        for a, d in enumerate((x - m, y - m, z)):
            nrm[..., a] = np.where(near, d / np.maximum(r, 1.0), 0.0)
        nrm[..., 2] = np.where(near, nrm[..., 2], np.where(z < n / 2, 1.0, -1.0))
        th = c["theta"] + 2.0 * jit()
        theta = np.where(near, th, 90.0)
        params = dict({**DROP, "sigma": 0.005}, theta_deg=th, **WETTED)
        s.update(dims=(n, n, n), solid=solid, normals=nrm, theta=theta, params=params,
                 init=dict(shape=0, center=(m + 0.2 * jit(), m + 0.2 * jit(), 50.0 * k + 0.2 * jit()),
                           R=20.0 * k * (1 + 0.02 * jit())))
        return s
    if kind == "slug":
        # Liquid between two plates, flat menisci relaxing to the angle.
        nx, ny, nz = c["nx"], c["H"] + 2, c["nz"]
        solid = np.zeros((nz, ny, nx), bool)
        solid[:, (0, ny - 1)] = True
        s.update(dims=(nx, ny, nz), solid=solid,
                 normals=_flat_normals(solid.shape, [(1, 1, 1.0), (1, ny - 2, -1.0)]),
                 params=dict(DROP, theta_deg=c["theta"] + 2.0 * jit(), **WETTED),
                 init=dict(shape=2, center=(nx / 2.0 - 0.5 + jit(), 0.0, 0.0),
                           R=nx / 6.0 * (1 + 0.05 * jit()), normal=(1.0, 0.0, 0.0)))
        return s
    if kind == "slit":
        # Plates over the middle of the box, liquid in the left reservoir.
        nx, ny, nz, res = c["nx"], c["ny"], c["nz"], c["reservoir"]
        solid = np.zeros((nz, ny, nx), bool)
        solid[:, (0, ny - 1), res:nx - res] = True
        s.update(dims=(nx, ny, nz), solid=solid,
                 params=dict(CAPILLARY, theta_deg=c["theta"] + 2.0 * jit(), **WETTED),
                 init=dict(shape=2, center=(res / 2.0 - 8.5 + 2.0 * jit(), 0.0, 0.0),
                           R=res / 2.0 - 8.0, normal=(1.0, 0.0, 0.0)))
        return s
    if kind == "duct":
        # A slug upstream of a square constriction in a square duct; pushed
        # by a body force, or by a pressure difference across open ends.
        w = c["w"]
        nx, ny = 4 * w, w + 2
        d = max(2, int(round(c["ratio"] * w)))
        lo = (ny - d) // 2
        solid = np.zeros((ny, ny, nx), bool)
        solid[(0, ny - 1), :] = True
        solid[:, (0, ny - 1)] = True
        block = np.ones((ny, ny), bool)
        block[lo:lo + d, lo:lo + d] = False
        solid[:, :, int(1.5 * w):int(2.5 * w)] |= block[:, :, None]
        th = c["theta"] + 2.0 * jit()
        pc = 4.0 * CAPILLARY["sigma"] * abs(math.cos(math.radians(th))) * (1.0 / d - 1.0 / w)
        pc = max(pc, 1e-4) * (0.8 + 0.1 * jit())
        params = dict(CAPILLARY, theta_deg=th, **WETTED)
        if not c.get("open"):
            params["Fex"] = (pc / nx, 0.0, 0.0)
        else:
            s["bounds"] = pc
        s.update(dims=(nx, ny, ny), solid=solid, params=params,
                 init=dict(shape=2, center=(0.75 * w - 0.5 + jit(), 0.0, 0.0), R=0.5 * w,
                           normal=(1.0, 0.0, 0.0)))
        return s
    if kind == "channel":
        # A drop on the axis of a square channel, carried by a body force.
        nx, ny = c["nx"], c["ny"]
        solid = np.zeros((ny, ny, nx), bool)
        solid[(0, ny - 1), :] = True
        solid[:, (0, ny - 1)] = True
        th = c["theta"] + 2.0 * jit()
        f = 28.45 * DROP["rho_L"] * DROP["nu_L"] * c["u"] / (ny - 2.0) ** 2
        m = (ny - 1) / 2.0
        s.update(dims=(nx, ny, ny), solid=solid,
                 params=dict({**DROP, "sigma": 0.005}, theta_deg=th, Fex=(f, 0.0, 0.0), **WETTED),
                 init=dict(shape=0, center=(nx / 4.0 + jit(), m + 0.3 * jit(), m + 0.3 * jit()),
                           R=c["R"] * (1 + 0.03 * jit())))
        return s
    raise ValueError(kind)


def _parts(c):
    """The single-lattice cases of a batch."""
    out = []
    for size in c["sizes"].split():
        if c["what"] == "duct":
            w = int(size)
            out.append(dict(kind="duct", w=w, ratio=0.4 + 0.3 * ((w * 7) % 11) / 10.0,
                            theta=95.0 + (w * 5) % 45, open=False, storage=c["storage"]))
        else:
            nx, ny = (int(v) for v in size.split("x"))
            out.append(dict(kind="channel", nx=nx, ny=ny, R=(0.3 + 0.01 * (nx % 13)) * ny,
                            theta=60.0 + nx % 60, u=1e-4 * (1 + nx % 10), storage=c["storage"]))
    return out


def _lattice(s, stream):
    nx, ny, nz = s["dims"]
    L = pflb.Lattice(nx, ny, nz, solid=s["solid"], wall_normal=s["normals"],
                     theta_cells=s["theta"], stream=stream, storage=s["storage"], **s["params"])
    i = s["init"]
    L.init_tanh(i["shape"], i["center"], i["R"], i.get("normal"))
    if s["bounds"] is not None:
        L.set_x_boundaries(dict(type="pressure", P=s["bounds"]), dict(type="pressure", P=0.0),
                           ramp_steps=100)
    return L


class _State:
    """A user's handles: lattices on a stream, and a batch where there is one."""

    def __init__(self, case, seed):
        self.case = case
        self.stream = torch.cuda.Stream()
        self.batch = None
        if case["kind"] == "batch":
            self.lattices = [_lattice(_setup(p, seed + 1000 * k), self.stream)
                             for k, p in enumerate(_parts(case))]
            self.batch = pflb.Batch(self.lattices, stream=self.stream)
        else:
            self.lattices = [_lattice(_setup(case, seed), self.stream)]
        if case.get("diag") or case["kind"] == "monitor":
            self.lattices[0].set_diag_every(1)

    def __del__(self):
        if self.batch is not None:
            self.batch.close()
        for L in self.lattices:
            L.close()


def prepare(case, seed):
    return _State(case, seed)


_TYPES = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.bfloat16,
          "bf16": torch.bfloat16}


def run(state):
    c = state.case
    t = _TYPES[c["storage"]]
    field = lambda L, f: torch.from_numpy(L.read(f)).to(t)  # noqa: E731
    if c["kind"] == "batch":
        state.batch.step(c["steps"], diag_last=True)
        return [field(L, "phi") for L in state.lattices]
    L = state.lattices[0]
    if c["kind"] == "monitor":
        mass = []
        for _ in range(c["steps"]):
            L.step(1)
            mass.append(L.last_diag()["mass"])
        return {"mass": torch.tensor(mass, dtype=torch.float32), "phi": field(L, "phi")}
    L.step(c["steps"])
    if c["storage"] == "fp64":
        return {f: field(L, f) for f in ("phi", "P", "ux", "uy", "uz")}
    out = {"phi": field(L, "phi")}
    if c["kind"] in ("drop", "sessile"):
        out["P"] = field(L, "P")
    if c.get("diag"):
        out["mass"] = L.last_diag()["mass"]
    return out


def work(case):
    """Bytes: every step reads and writes the 38 populations of each fluid
    cell once (16-bit storage: 39) and reads its flag; each field read back
    is written once.  Operations: about 700 per fluid cell and step."""
    b = total = flops = 0
    per = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}[case["storage"]]
    slots = 39 if per == 2 else 38
    for c in (_parts(case) if case["kind"] == "batch" else [case]):
        if c["kind"] in ("drop", "monitor"):
            fluid = total = c["nx"] * c["ny"] * c["nz"]
        elif c["kind"] == "sessile":
            total = c["n"] ** 3
            fluid = total - 2 * c["n"] ** 2 - int(2.0 / 3.0 * math.pi * (30.0 * c["n"] / 128) ** 3)
        elif c["kind"] == "slug":
            total = c["nx"] * (c["H"] + 2) * c["nz"]
            fluid = c["nx"] * c["H"] * c["nz"]
        elif c["kind"] == "slit":
            total = c["nx"] * c["ny"] * c["nz"]
            fluid = total - 2 * c["nz"] * (c["nx"] - 2 * c["reservoir"])
        elif c["kind"] == "duct":
            w = c["w"]
            d = max(2, int(round(c["ratio"] * w)))
            total = 4 * w * (w + 2) ** 2
            inside = int(2.5 * w) - int(1.5 * w)
            fluid = (4 * w - inside) * w * w + inside * d * d
        else:
            total = c["nx"] * c["ny"] ** 2
            fluid = c["nx"] * (c["ny"] - 2) ** 2
        fields = 5 if per == 8 else 2 if c["kind"] in ("drop", "sessile") else 1
        b += case["steps"] * fluid * (2 * slots * per + 1) + fields * total * 8
        flops += case["steps"] * fluid * 700
    return {"bytes": b, "flops": flops}


# ------------------------------------------------------- 64-bit reference

_C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
      (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
      (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
_WT = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12
_OPP = [_C.index(tuple(-v for v in c)) for c in _C]


def _at(v, c):
    """v at x + c (arrays are [z, y, x], periodic)."""
    return torch.roll(v, shifts=(-c[2], -c[1], -c[0]), dims=(0, 1, 2)) if any(c) else v


class _Exact:
    """The method in 64 bits on whole arrays."""

    GAMMA, PHI_HI, PHI_LO, D, EPS = -22.5, 0.8, 0.2, 1e-4, 1e-10
    BAND_LO, BAND_HI, F_MID, F_WIDTH = 0.5, 0.95, 0.1, 0.001

    def __init__(self, s):
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.p = p = s["params"]
        self.F = p.get("Fex", (0.0, 0.0, 0.0))
        nx, ny, nz = s["dims"]
        self.shape = (nz, ny, nx)
        f8 = dict(dtype=torch.float64, device=self.dev)
        solid = s["solid"]
        self.solid = torch.zeros(self.shape, dtype=torch.bool, device=self.dev) if solid is None \
            else torch.from_numpy(np.ascontiguousarray(solid)).to(self.dev)
        self.walls = bool(self.solid.any())
        self.bounds, self.t = s["bounds"], 0
        self.live = ~self.solid
        i = s["init"]
        ax = [torch.arange(n, **f8) for n in (nx, ny, nz)]
        d = [ax[a] - i["center"][a] for a in range(3)]
        d = [v - n * torch.round(v / n) for v, n in zip(d, (nx, ny, nz))]
        dx, dy, dz = d[0][None, None, :], d[1][None, :, None], d[2][:, None, None]
        if i["shape"] == 0:
            arg = i["R"] - torch.sqrt(dx * dx + dy * dy + dz * dz)
        else:
            n = i["normal"]
            arg = i["R"] - (dx * n[0] + dy * n[1] + dz * n[2]).abs() + torch.zeros(self.shape, **f8)
        phi = 0.5 * (1.0 + torch.tanh(2.0 * arg / p["W"]))
        if self.walls:
            self._wall_setup(s, phi, f8)
        val = [phi] + [torch.where(self.lm[k], phi, _at(phi, _C[k])) if self.walls
                       else _at(phi, _C[k]) for k in range(1, 19)]
        gx, gy, gz, lap = self._stencil(val)
        mu = self._mu(phi, lap)
        thn = self._theta(phi, gx, gy, gz, lap)
        self.h, self.g = [None] * 19, []
        for k, (c, w) in enumerate(zip(_C, _WT)):
            cg = c[0] * gx + c[1] * gy + c[2] * gz
            cf = sum(a * b for a, b in zip(c, self.F))
            self.g.append(torch.where(self.live, -1.5 * w * (mu * cg + cf), 0.0))
            self.h[k] = torch.where(self.live, w * phi + w * thn * cg, 0.0)
        self.h[0] = torch.where(self.live, phi, 0.0) - sum(self.h[1:])

    def _wall_setup(self, s, phi, f8):
        self.lm = [None] + [_at(self.solid, c) & self.live for c in _C[1:]]
        self.wall = torch.stack(self.lm[1:]).any(0)
        self.ghost = [None] + [torch.where(m, phi, 0.0) for m in self.lm[1:]]
        if s["normals"] is not None:
            n = torch.from_numpy(np.ascontiguousarray(s["normals"])).to(self.dev)
            n = [n[..., a].reshape(self.shape).clone() for a in range(3)]
        else:
            n = [torch.zeros(self.shape, **f8) for _ in range(3)]
            for k in range(1, 19):
                for a in range(3):
                    if _C[k][a]:
                        n[a] -= _WT[k] * _C[k][a] * self.lm[k].double()
            nn = torch.sqrt(n[0] ** 2 + n[1] ** 2 + n[2] ** 2)
            nn = torch.where(nn > 0, nn, 1.0)
            n = [v / nn for v in n]
        th = s["params"]["theta_deg"] if s["theta"] is None else s["theta"]
        th = torch.as_tensor(th, dtype=torch.float64, device=self.dev) * (math.pi / 180.0)
        self.n, self.ct, self.st = n, torch.cos(th), torch.sin(th)

    def _stencil(self, v):
        gx, gy, gz = 0.0, 0.0, 0.0
        lap = -6.0 * (1.0 - _WT[0]) * v[0]
        for k in range(1, 19):
            c, w = _C[k], _WT[k]
            if c[0]:
                gx = gx + 3.0 * w * c[0] * v[k]
            if c[1]:
                gy = gy + 3.0 * w * c[1] * v[k]
            if c[2]:
                gz = gz + 3.0 * w * c[2] * v[k]
            lap = lap + 6.0 * w * v[k]
        return gx, gy, gz, lap

    def _mu(self, phi, lap):
        p = self.p
        return 48.0 * p["sigma"] / p["W"] * phi * (phi - 1.0) * (phi - 0.5) \
            - 1.5 * p["sigma"] * p["W"] * lap

    def _theta(self, phi, gx, gy, gz, lap):
        """theta + delta theta over |grad phi| (Eqs. 3-4)."""
        p = self.p
        k = 3.0 * p["M"] / p["W"]
        gn = torch.sqrt(gx * gx + gy * gy + gz * gz)
        cl = lambda v: torch.clamp(v / self.D, 0.0, 1.0)  # noqa: E731
        y1 = torch.minimum(cl(phi - self.PHI_HI), cl(1.0 - phi))
        y2 = torch.minimum(cl(phi), cl(self.PHI_LO - phi))
        sg = lap / (lap.abs() + self.EPS)
        th = k * (1.0 - 4.0 * (phi - 0.5) ** 2)
        if p["mobility_corr"]:
            th = th + self.GAMMA * k * gn * ((1.0 + sg) * y1 + (1.0 - sg) * y2)
        return th / (gn + self.EPS)

    def _boundary(self):
        """Boundary states (phi, P, u) of the open x planes: given pressure,
        the rest from the adjacent cell."""
        f = min(1.0, self.t / 100.0)
        out = []
        for at, P in ((1, self.bounds * f), (self.shape[2] - 2, 0.0)):
            ok = self.live[:, :, at]
            ph = torch.where(ok, sum(h[:, :, at] for h in self.h), 0.0)
            rho = self.p["rho_L"] + ph * (self.p["rho_H"] - self.p["rho_L"])
            u = []
            for a in range(3):
                m = sum(c[a] * g[:, :, at] for c, g in zip(_C, self.g) if c[a])
                u.append(torch.where(ok, (m + 0.5 * self.F[a]) / rho, 0.0))
            out.append((ph, torch.full_like(ph, P), u, rho))
        return out

    def fields(self, advance=False):
        """Macroscopic fields of the present state; with advance, also the
        step (Eqs. 1-11 and the streaming with wall reflection)."""
        p, F = self.p, self.F
        rho_d = p["rho_H"] - p["rho_L"]
        phi = torch.where(self.live, sum(self.h), 0.0)
        bc = self._boundary() if self.bounds is not None else None
        planes = (0, self.shape[2] - 1)
        if bc:
            for x, b in zip(planes, bc):
                phi[:, :, x] = torch.where(self.live[:, :, x], b[0], 0.0)
        val = [phi] + [_at(phi, c) for c in _C[1:]]
        if self.walls:
            for k in range(1, 19):
                val[k] = torch.where(self.lm[k], self.ghost[k], val[k])
            gx, gy, gz, _ = self._stencil(val)
            n = self.n
            gn = gx * n[0] + gy * n[1] + gz * n[2]
            t = [gx - gn * n[0], gy - gn * n[1], gz - gn * n[2]]
            t2 = t[0] ** 2 + t[1] ** 2 + t[2] ** 2
            inv = torch.where(t2 >= 1e-20, 1.0 / torch.sqrt(torch.clamp(t2, min=1e-300)), 0.0)
            w = [-self.ct * n[a] + self.st * t[a] * inv for a in range(3)]
            sm = torch.clamp(2.0 * phi - 1.0, -1.0, 1.0)
            new = [None]
            for k in range(1, 19):
                c = _C[k]
                tb = torch.tanh(2.0 / p["W"] * (w[0] * c[0] + w[1] * c[1] + w[2] * c[2]))
                fresh = 0.5 * (1.0 + (sm + tb) / (1.0 + sm * tb))
                gk = torch.where(self.lm[k],
                                 p["blend"] * self.ghost[k] + (1.0 - p["blend"]) * fresh, 0.0)
                if bc:  # boundary cells keep theirs
                    for x in planes:
                        gk[:, :, x] = self.ghost[k][:, :, x]
                new.append(gk)
                val[k] = torch.where(self.lm[k], gk, val[k])
        gx, gy, gz, lap = self._stencil(val)
        mu = self._mu(phi, lap)
        rho = p["rho_L"] + phi * rho_d
        u = []
        for a, gr in enumerate((gx, gy, gz)):
            j = sum(c[a] * g for c, g in zip(_C, self.g) if c[a])
            u.append((j + 0.5 * (mu * gr + F[a])) / rho)
        ug = u[0] * gx + u[1] * gy + u[2] * gz
        P = sum(self.g) / 3.0 + rho_d / 6.0 * ug
        if bc:
            for x, b in zip(planes, bc):
                P[:, :, x] = b[1]
        if not advance:
            return dict(phi=phi, P=torch.where(self.live, P, 0.0),
                        **{k: torch.where(self.live, v, 0.0) for k, v in zip(("ux", "uy", "uz"), u)})
        thn = self._theta(phi, gx, gy, gz, lap)
        om = 1.0 / (3.0 * p["M"] + 0.5)
        uu = 1.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        uF = sum(a * b for a, b in zip(u, F))
        hs, gs, pi = [None] * 19, [None] * 19, [[0.0] * 3 for _ in range(3)]
        rest = phi.clone()
        for k, (c, w) in enumerate(zip(_C, _WT)):
            cu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2]
            cgr = c[0] * gx + c[1] * gy + c[2] * gz
            dG = w * (cu * (3.0 + 4.5 * cu) - uu)
            if k:
                hs[k] = self.h[k] + om * (phi * (w + dG) + thn * w * cgr - self.h[k])
                rest -= hs[k]
            K = (dG * rho_d + (w + dG) * 3.0 * mu) * (cgr - ug)
            if any(F):
                K = K + 3.0 * (w + dG) * (sum(a * b for a, b in zip(c, F)) - uF)
            b = 3.0 * w * P + rho * dG + 0.5 * K
            neq = self.g[k] - b + K
            gs[k] = b
            for i in range(3):
                for j in range(i, 3):
                    if c[i] * c[j]:
                        pi[i][j] = pi[i][j] + c[i] * c[j] * neq
        hs[0] = rest
        Fp = phi if p["F_mode"] == 0 else \
            0.5 * (torch.tanh((phi - self.F_MID) / self.F_WIDTH) + 1.0)
        tau = (1.0 - Fp) * (3.0 * p["nu_L"] + 0.5) + Fp * (3.0 * p["nu_H"] + 0.5)
        f = 4.5 * (1.0 - 1.0 / tau)
        tr = (pi[0][0] + pi[1][1] + pi[2][2]) / 3.0
        for k, (c, w) in enumerate(zip(_C, _WT)):
            cc = -tr
            for i in range(3):
                for j in range(i, 3):
                    if c[i] * c[j]:
                        cc = cc + (1.0 if i == j else 2.0) * c[i] * c[j] * pi[i][j]
            gs[k] = gs[k] + f * w * cc
        if bc:  # boundary cells: equilibria at the boundary state
            for x, (ph, Pb, ub, _) in zip(planes, bc):
                rb = p["rho_L"] + ph * rho_d
                ub2 = 1.5 * (ub[0] ** 2 + ub[1] ** 2 + ub[2] ** 2)
                for k, (c, w) in enumerate(zip(_C, _WT)):
                    cu = c[0] * ub[0] + c[1] * ub[1] + c[2] * ub[2]
                    dG = w * (cu * (3.0 + 4.5 * cu) - ub2)
                    hs[k][:, :, x] = ph * (w + dG)
                    gs[k][:, :, x] = 3.0 * w * Pb + rb * dG
        self._stream(phi, hs, gs, planes if bc else ())
        if self.walls:
            self.ghost = new
        self.t += 1
        return None

    def _stream(self, phi, hs, gs, open_planes):
        slip = self.walls and self.p["free_slip"]
        if slip:
            band = (phi >= self.BAND_LO) & (phi <= self.BAND_HI) & self.live
            own = band.clone()
            for x in open_planes:
                own[:, :, x] = False
        h, g = [], []
        for k, c in enumerate(_C):
            o = _OPP[k]
            back = tuple(-v for v in c)
            hk, gk = _at(hs[k], back), _at(gs[k], back)
            if k and self.walls:
                hk = torch.where(self.lm[o], hs[o], hk)
                refl = gs[o]
                axes = [a for a in range(3) if c[a]]
                if slip and len(axes) == 2:
                    # link o = (along a, along b): flat wall across a, fluid
                    # neighbour y = x + o_b, or the other way round
                    co = _C[o]
                    e = [tuple(co[a] if a == q else 0 for a in range(3)) for q in axes]
                    sa, sb = (self.lm[_C.index(v)] for v in e)
                    for into, along, hit in ((0, 1, sa & ~sb), (1, 0, sb & ~sa)):
                        m = _C.index(tuple(-v if a == axes[into] else v for a, v in enumerate(c)))
                        yes = hit & own & _at(own, e[along]) & _at(self.live, e[along])
                        refl = torch.where(yes, _at(gs[m], e[along]), refl)
                gk = torch.where(self.lm[o], refl, gk)
            h.append(torch.where(self.live, hk, 0.0) if self.walls else hk)
            g.append(torch.where(self.live, gk, 0.0) if self.walls else gk)
        self.h, self.g = h, g

    def mass(self):
        return float(torch.where(self.live, sum(self.h), 0.0).sum())


def exact(case, seed):
    flat = lambda v: v.reshape(-1).cpu()  # noqa: E731
    with torch.no_grad():
        if case["kind"] == "batch":
            out = []
            for k, part in enumerate(_parts(case)):
                e = _Exact(_setup(part, seed + 1000 * k))
                for _ in range(case["steps"]):
                    e.fields(advance=True)
                out.append(flat(e.fields()["phi"]))
            return out
        e = _Exact(_setup(case, seed))
        mass = []
        for _ in range(case["steps"]):
            if case["kind"] == "monitor" or case.get("diag"):
                mass.append(e.mass())
            e.fields(advance=True)
        f = e.fields()
        if case["kind"] == "monitor":
            return {"mass": torch.tensor(mass, dtype=torch.float64), "phi": flat(f["phi"])}
        if case["storage"] == "fp64":
            return {k: flat(f[k]) for k in ("phi", "P", "ux", "uy", "uz")}
        out = {"phi": flat(f["phi"])}
        if case["kind"] in ("drop", "sessile"):
            out["P"] = flat(f["P"])
        if case.get("diag"):
            out["mass"] = torch.tensor(mass[-1], dtype=torch.float64)
        return out
