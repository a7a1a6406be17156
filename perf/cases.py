"""Timed workloads of the library: what a program that uses it has it do.

A case is one simulation (or one batch, or one gradient) in the state that a
program holds: a handle, its initial fields on the GPU and the tensors that
receive the fields.  One pass advances it and reads the macroscopic fields,
through the public entry points (``Lattice``, ``Lattice1``, ``Lattice3``,
``Batch``, ``Adjoint`` and, for fields kept on the device in one and three
dimensions, the C calls ``rlbm1_moments`` and ``rlbm3_moments``).  The
populations come back too wherever a call gives their device buffer
(``rlbm_buffers``).  Sizes are those of the benchmark and of the tests, and
odd ones between them.

``exact`` repeats a pass in 64 bits from the definitions (Sec. 4-6.2, App. B,
App. H of arXiv:1909.04502) with torch alone.
"""
import ctypes
import decimal
import itertools
import math

import numpy as np
import torch

from paper_1909_04502_gb300 import rlbm

# Stencils of the massive gases: FS generators and v0 by (m, order), those that
# the library picks by itself (Sec. 5.3 example, App. H columns), and at
# (15, 3) the 45-vector stencil of the paper's performance table.
STENCILS = {
    (1.0, 2): (((0, 0), (3, 3), (4, 2), (4, 3), (5, 0), (5, 1)), 0.19518481632598073),
    (5.0, 2): (((0, 0), (1, 0), (1, 1), (2, 1), (2, 2), (3, 1)), 0.27267827861986776),
    (10.0, 2): (((0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (2, 2)), 0.3068076411246804),
    (1.5, 3): (((0, 0), (1, 1), (4, 2), (5, 4), (5, 5), (6, 2), (6, 3), (6, 4), (7, 1), (7, 2)), 0.13615895941527134),
    (5.0, 3): (((0, 0), (1, 0), (2, 0), (2, 2), (3, 0), (3, 2), (3, 3), (4, 0), (4, 1), (4, 2)), 0.21986232000710254),
    (10.0, 3): (((0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (3, 1), (3, 2), (3, 3), (4, 0), (4, 2)), 0.18996238579159672),
    (15.0, 3): (((0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (2, 2), (3, 0), (3, 2), (3, 3), (4, 0)), 0.1970272956492884),
}
POPULATIONS = {(0.0, 2): 28, (0.0, 3): 44, (1.0, 2): 33, (5.0, 2): 29, (10.0, 2): 25, (1.5, 3): 65, (5.0, 3): 49,
               (10.0, 3): 53, (15.0, 3): 45}
POPULATIONS3 = {2: 78, 3: 288}


def listed():
    return [
        # the shock tube of the 1-d validation and of the viscosity calibration, from its
        # initial state to the fields: the smallest grid, where launches and latency count
        {"name": "tube_1024", "kind": "flow", "flow": "tube", "nx": 1024, "ny": 1, "m": 0.0, "order": 2,
         "precision": "fp32", "stream": "onlattice", "tau": 0.0, "steps": 40},
        # a calibration sweep of small shear waves of three masses, stepped together
        {"name": "sweep_24", "kind": "batch", "count": 24, "side_lo": 64, "side_hi": 256, "steps": 10},
        # the benchmark's headline: Taylor-Green vortex, off-lattice streaming
        {"name": "vortex_512_bilinear", "kind": "flow", "flow": "vortex", "nx": 512, "ny": 512, "m": 0.0, "order": 2,
         "precision": "fp32", "stream": "bilinear", "tau": 1.0, "steps": 20},
        # the same gas in double precision on a grid that no tile divides
        {"name": "vortex_517x333_fp64", "kind": "flow", "flow": "vortex", "nx": 517, "ny": 333, "m": 0.0, "order": 2,
         "precision": "fp64", "stream": "onlattice", "tau": 0.9, "steps": 8},
        # the paper's performance table: third order, zeta = 5, double precision
        {"name": "vortex_512_order3_fp64", "kind": "flow", "flow": "vortex", "nx": 512, "ny": 512, "m": 5.0,
         "order": 3, "precision": "fp64", "stream": "onlattice", "tau": 1.0, "steps": 4},
        # the Kelvin-Helmholtz layer at its full size
        {"name": "layer_2048_order3", "kind": "flow", "flow": "layer", "nx": 2048, "ny": 2048, "m": 1.5, "order": 3,
         "precision": "fp32", "stream": "onlattice", "tau": 0.85, "steps": 6},
        # forced channel between equilibrium walls
        {"name": "channel_4096x1024", "kind": "flow", "flow": "channel", "nx": 4096, "ny": 1024, "m": 5.0, "order": 2,
         "precision": "fp32", "stream": "onlattice", "tau": 1.0, "steps": 6},
        # the (1+1)-d gas in the precision that Lattice1 takes by default
        {"name": "wave_2e24_fp64", "kind": "wave", "nx": 1 << 24, "order": 3, "precision": "fp64", "tau": 0.9,
         "steps": 4},
        # the (3+1)-d vortex: second order at full size with FP32 storage,
        {"name": "vortex3_192", "kind": "flow3", "nx": 192, "ny": 192, "nz": 192, "order": 2, "precision": "fp32",
         "tau": 0.8, "steps": 10},
        # second order in the default precision on a ragged box,
        {"name": "vortex3_101x75x66_fp64", "kind": "flow3", "nx": 101, "ny": 75, "nz": 66, "order": 2,
         "precision": "fp64", "tau": 0.8, "steps": 5},
        # and third order in double precision on the slab of the paper's Table 2
        {"name": "vortex3_192x192x6_order3_fp64", "kind": "flow3", "nx": 192, "ny": 192, "nz": 6, "order": 3,
         "precision": "fp64", "tau": 0.6, "steps": 5},
        # gradient of a run with respect to its relaxation times and initial flow
        {"name": "adjoint_512", "kind": "adjoint", "nx": 512, "ny": 512, "precision": "fp32", "stream": "onlattice",
         "steps": 96, "every": 32},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["flow"] * 6 + ["flow3"] * 3 + ["wave", "batch", "adjoint"])
    tau = round(rng.uniform(0.7, 1.5), 3)
    prec = rng.choice(["fp32", "fp64"])
    if kind == "flow3":
        order = rng.choice([2, 2, 3])
        top = {(2, "fp32"): 160, (2, "fp64"): 96, (3, "fp32"): 72, (3, "fp64"): 60}[order, prec]
        return {"kind": kind, "nx": _log(rng, 16, top), "ny": _log(rng, 16, top), "nz": _log(rng, 6, top),
                "order": order, "precision": prec, "tau": tau, "steps": rng.randint(3, 8)}
    if kind == "wave":
        return {"kind": kind, "nx": _log(rng, 1000, 1 << (23 if prec == "fp32" else 21)), "order": rng.randint(2, 5),
                "precision": prec, "tau": tau, "steps": rng.randint(3, 8)}
    if kind == "batch":
        lo = rng.randint(32, 128)
        return {"kind": kind, "count": rng.randint(3, 32), "side_lo": lo, "side_hi": lo + rng.randint(1, 200),
                "steps": rng.randint(4, 16)}
    if kind == "adjoint":
        top = 500 if prec == "fp32" else 200
        return {"kind": kind, "nx": _log(rng, 32, top), "ny": _log(rng, 32, top), "precision": prec,
                "stream": rng.choice(["onlattice", "bilinear"]), "steps": rng.randint(8, 40),
                "every": rng.randint(4, 16)}
    flow = rng.choice(["tube", "vortex", "vortex", "vortex", "layer", "channel"])
    if flow == "tube":
        return {"kind": kind, "flow": flow, "nx": _log(rng, 200, 200000), "ny": 1, "m": 0.0, "order": 2,
                "precision": prec, "stream": "onlattice", "tau": 0.0, "steps": rng.randint(10, 40)}
    m, order = rng.choice([(0.0, 2), (0.0, 2), (0.0, 3)] + sorted(STENCILS))
    stream = "onlattice"
    if flow == "vortex" and rng.random() < 0.3:
        stream = "bilinear"
    if flow == "layer":
        m, order = 1.5, 3
    if flow == "channel":
        m, order = rng.choice([(1.0, 2), (5.0, 2), (5.0, 3)])
    top = 1600 if prec == "fp32" else 700
    return {"kind": kind, "flow": flow, "nx": _log(rng, 40, top), "ny": _log(rng, 40, top), "m": m, "order": order,
            "precision": prec, "stream": stream, "tau": 0.85 if flow == "layer" else tau,
            "steps": rng.randint(3, 10)}


# ---------------------------------------------------------------------------
# Initial states: what the flow is at the start, from the seed alone.
# ---------------------------------------------------------------------------

KAPPA, ETA_S = 15.79, 0.1      # the tube's hbar / (k_B T0 dt) and eta / s
LAM = 1.0                      # cells per step of the off-lattice streaming
GRAVITY = (0.0, 1e-6)


def _grid(*sides):
    """Coordinates in [0, 2 pi), x first, each shaped like the (z,) y, x fields."""
    axes = [2 * math.pi / n * torch.arange(n, device="cuda", dtype=torch.float64) for n in reversed(sides)]
    return list(reversed(torch.meshgrid(*axes, indexing="ij")))


def _fields2(flow, nx, ny, seed, T0=1.0):
    rng = np.random.RandomState(seed % (1 << 31))
    a, b, c, d = rng.uniform(0, 2 * math.pi, 4)
    X, Y = _grid(nx, ny)
    one = torch.ones_like(X)
    if flow == "tube":
        left = torch.arange(nx, device="cuda").expand(ny, nx) < nx // 2 + int(rng.randint(-nx // 50, nx // 50 + 1))
        nr, tr = rng.uniform(0.45, 0.55), rng.uniform(0.75, 0.85)
        return (torch.where(left, one, nr * one), 0 * one, 0 * one, torch.where(left, one, tr * one))
    if flow == "shear":
        return (one.clone(), 0 * one, 0.05 * torch.sin(X + a), one.clone())
    if flow == "layer":
        y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None].expand(ny, nx)
        w = 20.0 * ny / 2048 + 2.0
        ux = 0.3 * (torch.tanh((y - ny / 4) / w) - torch.tanh((y - 3 * ny / 4) / w) - 1.0)
        gen = torch.Generator(device="cuda").manual_seed(int(seed))
        uy = 1e-3 * (2 * torch.rand(ny, nx, device="cuda", dtype=torch.float64, generator=gen) - 1)
        return (one.clone(), ux.contiguous(), uy, T0 * one)
    n = 1.0 + 0.02 * torch.cos(X + b) * torch.cos(Y + c)
    T = T0 * (1.0 + 0.02 * torch.sin(X + d) * torch.cos(Y + a))
    if flow == "channel":
        x = torch.arange(nx, device="cuda", dtype=torch.float64).expand(ny, nx) / max(nx - 1, 1)
        return (n, 0.01 * torch.sin(X) * torch.sin(Y + a), 0.2 * x * (1 - x) + 0.005 * torch.cos(X + b), T)
    return (n, 0.1 * torch.cos(X + a) * torch.sin(Y + b), -0.1 * torch.cos(Y + b) * torch.sin(X + a), T)


def _fields3(nx, ny, nz, seed):
    a, b, c = np.random.RandomState(seed % (1 << 31)).uniform(0, 2 * math.pi, 3)
    X, Y, Z = _grid(nx, ny, nz)
    n = 1.0 + 0.02 * torch.cos(X + b) * torch.cos(Z + c)
    T = 1.0 + 0.02 * torch.sin(Y + c) * torch.cos(X + a)
    return (n, 0.15 * torch.cos(X + a) * torch.sin(Y + b), -0.15 * torch.cos(Y + b) * torch.sin(X + a),
            0.02 * torch.sin(Z + a) * torch.cos(X + c), T)


def _fields1(nx, seed):
    a, b = np.random.RandomState(seed % (1 << 31)).uniform(0, 2 * math.pi, 2)
    x = 2 * math.pi / nx * torch.arange(nx, device="cuda", dtype=torch.float64)
    return 1 + 0.1 * torch.sin(x + a), 0.2 * torch.cos(x + b), 1 + 0.1 * torch.cos(x + a)


def _sweep(c, seed):
    """Sides, relaxation times and masses of a sweep's instances (the masses in turn)."""
    rng = np.random.RandomState(1909)      # the sides are the case's, so that the work does not depend on the seed
    sides = rng.randint(c["side_lo"], c["side_hi"] + 1, c["count"])
    taus = np.random.RandomState(seed % (1 << 31)).uniform(0.6, 2.0, c["count"])
    return [(int(s), float(t), (0.0, 1.0, 10.0)[i % 3]) for i, (s, t) in enumerate(zip(sides, taus))]


def _stencil(m, order):
    if m == 0.0:
        return {}
    groups, v0 = STENCILS[(m, order)]
    return {"groups": groups, "v0": v0}


def _options(c):
    """Keyword arguments of Lattice for a flow case."""
    o = dict(m=c["m"], order=c["order"], precision=c["precision"], stream=c["stream"], tau=c["tau"])
    if c["flow"] != "channel":      # the channel takes the stencil that the library picks (the same)
        o.update(_stencil(c["m"], c["order"]))
    if c["stream"] == "bilinear":
        o["lam"] = LAM
    if c["flow"] == "tube":
        o.update(d=1, boundary="freeflow_x", tau=1.0, tau_mode="eta_over_s", eta_over_s=ETA_S, kappa=KAPPA)
    elif c["flow"] == "layer":
        o["T_ref"] = 1.5
    elif c["flow"] == "channel":
        o.update(boundary="eqwall_x", g=GRAVITY)
    return o


def _T0(c):
    return 1.5 if c.get("flow") == "layer" else 1.0


# ---------------------------------------------------------------------------
# A pass
# ---------------------------------------------------------------------------


class _Memory:
    """Device memory of `owner` (a Lattice or a Batch) for torch, which holds this object as long as a tensor is on
    the memory: the handle outlives the tensors."""

    def __init__(self, owner, ptr, nbytes):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": (nbytes,), "typestr": "|u1", "data": (ptr, False), "version": 3,
                                         "strides": None}


def _views(lat, owner=None):
    """The interior of a handle's two population buffers as (Q, ny, nx) tensors, by device pointer."""
    cur, prev, elem, plane, (pitch, hx, hy, px) = lat.buffers()
    kind = torch.float32 if elem == 4 else torch.float64
    out = {}
    for ptr in (cur, prev):
        raw = torch.as_tensor(_Memory(owner or lat, ptr, lat.Q * plane * elem), device="cuda").view(kind)
        out[ptr] = raw.as_strided((lat.Q, lat.ny, lat.nx), (plane, pitch, 1), hy * pitch + px)
    return out


PLANES2 = (("n", 1), ("ux", 1), ("uy", 1), ("T", 1), ("eps", 1), ("N", 3), ("Tab", 6))
PLANES3 = (("n", 1), ("ux", 1), ("uy", 1), ("uz", 1), ("T", 1), ("eps", 1))
PLANES1 = (("n", 1), ("ux", 1), ("T", 1), ("eps", 1), ("N0", 1), ("Nx", 1), ("T00", 1), ("T0x", 1))


class _Fields:
    """The tensors that receive the fields (doubles, as the library gives them), and the snapshot a program keeps: the
    same tensors, or 32-bit copies where the handle stores its state in 32 bits, which resolve no more."""

    def __init__(self, planes, shape, precision):
        self.all = torch.empty((sum(k for _, k in planes),) + shape, device="cuda", dtype=torch.float64)
        self.out = self._named(self.all, planes)
        self.copy = torch.empty_like(self.all, dtype=torch.float32) if precision == "fp32" else None
        self.kept = self.out if self.copy is None else self._named(self.copy, planes)

    @staticmethod
    def _named(a, planes):
        named, at = {}, 0
        for name, k in planes:
            named[name] = a[at] if k == 1 else a[at:at + k]
            at += k
        return named

    def snapshot(self):
        if self.copy is not None:
            self.copy.copy_(self.all)
        return self.kept


def prepare(case, seed):
    c, k = case, case["kind"]
    if k == "flow":
        lat = rlbm.Lattice(c["nx"], c["ny"], **_options(c))
        f = [a.contiguous() for a in _fields2(c["flow"], c["nx"], c["ny"], seed, _T0(c))]
        lat.init(*f)
        # a shock tube's program reads no transverse velocity: it is the rounding's
        planes = [p for p in PLANES2 if p[0] != "uy" or c["flow"] != "tube"]
        return {"case": c, "lat": lat, "fields": f, "out": _Fields(planes, (c["ny"], c["nx"]), c["precision"]),
                "views": _views(lat)}
    if k == "flow3":
        lat = rlbm.Lattice3(c["nx"], c["ny"], c["nz"], tau=c["tau"], precision=c["precision"], order=c["order"])
        f = [a.contiguous() for a in _fields3(c["nx"], c["ny"], c["nz"], seed)]
        lat.init(*f)
        return {"case": c, "lat": lat, "fields": f,
                "out": _Fields(PLANES3, (c["nz"], c["ny"], c["nx"]), c["precision"])}
    if k == "wave":
        lat = rlbm.Lattice1(c["nx"], order=c["order"], tau=c["tau"], precision=c["precision"])
        f = _fields1(c["nx"], seed)
        lat.init(*f)
        return {"case": c, "lat": lat, "fields": f, "out": _Fields(PLANES1, (c["nx"],), c["precision"])}
    if k == "batch":
        runs = _sweep(c, seed)
        batch = rlbm.Batch([dict(nx=s, ny=s, tau=t, m=m, precision="fp32", **_stencil(m, 2)) for s, t, m in runs])
        batch.tune(trial_steps=2)
        fields = []
        for i, (s, _, _) in enumerate(runs):
            fields.append([a.contiguous() for a in _fields2("shear", s, s, seed + i)])
            batch[i].init(*fields[-1])
        return {"case": c, "batch": batch, "fields": fields, "views": [_views(lat, batch) for lat in batch.instances]}
    lat = rlbm.Lattice(c["nx"], c["ny"], precision=c["precision"], stream=c["stream"], tau=1.0,
                       **({"lam": LAM} if c["stream"] == "bilinear" else {}))
    f = [a.contiguous() for a in _fields2("shear", c["nx"], c["ny"], seed)]
    target = _target(c, f)
    return {"case": c, "lat": lat, "adjoint": rlbm.Adjoint(lat, c["steps"], c["every"]), "fields": f, "target": target,
            "loss": torch.empty(1, device="cuda", dtype=torch.float64),
            "out": _Fields((("tau", 1), ("ux0", 1), ("uy0", 1)), (c["ny"], c["nx"]), c["precision"])}


def _target(c, f):
    X, Y = _grid(c["nx"], c["ny"])
    return (0.01 * torch.cos(Y)).contiguous(), (0.8 * f[2] + 0.01 * torch.cos(X)).contiguous()


def run(state):
    c = state["case"]
    k = c["kind"]
    if k == "flow":
        lat = state["lat"]
        if c["flow"] == "tube":
            lat.init(*state["fields"])
        lat.step(c["steps"])
        lat.moments(full=True, out=state["out"].out)
        return {"fields": state["out"].snapshot(), "f": state["views"][lat.buffers()[0]]}
    if k == "flow3":
        state["lat"].step(c["steps"])
        _check(rlbm.lib().rlbm3_moments(state["lat"].h, ctypes.c_void_p(state["out"].all.data_ptr()), 1))
        return state["out"].snapshot()
    if k == "wave":
        state["lat"].step(c["steps"])
        _check(rlbm.lib().rlbm1_moments(state["lat"].h, ctypes.c_void_p(state["out"].all.data_ptr()), 1))
        return state["out"].snapshot()
    if k == "batch":
        state["batch"].step(c["steps"])
        return [v[lat.buffers()[0]] for v, lat in zip(state["views"], state["batch"].instances)]
    state["adjoint"].forward(*state["fields"])
    state["adjoint"].backward(*state["target"], out={"loss": state["loss"], **state["out"].out})
    return state["out"].snapshot()


def _check(rc):
    if rc != rlbm.RLBM_OK:
        raise RuntimeError("the library returned %d" % rc)


def work(case):
    """Every step reads and writes each population once (the states that matter exceed the chip's caches by far); the
    fields read them once more and are written once.  Operations per cell and step: the moment sums, the
    equilibrium's contraction and the relaxation."""
    c, k = case, case["kind"]
    b = 4 if c.get("precision", "fp32") == "fp32" else 8
    if k == "batch":
        by = fl = 0
        for s, _, m in _sweep(c, 0):
            by += c["steps"] * 2 * POPULATIONS[(m, 2)] * 4 * s * s
            fl += c["steps"] * POPULATIONS[(m, 2)] * 2 * (9 + 9 + 3) * s * s
        return {"bytes": by, "flops": fl}
    if k == "wave":
        q, K, sums, fields, cells = 2 * c["order"], 2 * c["order"], 4, 8, c["nx"]
    elif k == "flow3":
        q, K, sums, fields = POPULATIONS3[c["order"]], 14 if c["order"] == 2 else 30, 14, 6
        cells = c["nx"] * c["ny"] * c["nz"]
    else:
        q = POPULATIONS[(c.get("m", 0.0), c.get("order", 2))]
        K, sums, fields, cells = 9 if c.get("order", 2) == 2 else 16, 9, 14, c["nx"] * c["ny"]
    step, flops = 2 * q * b, q * 2 * (sums + K + 3)
    if k == "adjoint":
        # forward; then per step the states again and the adjoint step (reads f, a; writes a; tau, its gradient)
        by = c["steps"] * (step + step + 3 * q * b + 24)
        return {"bytes": cells * (by + 9 * 8), "flops": cells * c["steps"] * 4 * flops}
    by = c["steps"] * step + q * b + 8 * fields
    if c.get("flow") == "tube":
        by += q * b + 4 * 8
    return {"bytes": cells * by, "flops": cells * (c["steps"] * flops + q * 2 * sums)}


# ---------------------------------------------------------------------------
# The same pass in 64 bits, from the definitions.
# ---------------------------------------------------------------------------

D = decimal.Decimal


def _solve(A, B):
    """A X = B in 60 digits (Gauss-Jordan with pivoting); B has several columns."""
    n = len(A)
    A = [list(r) + list(b) for r, b in zip(A, B)]
    for j in range(n):
        p = max(range(j, n), key=lambda i: abs(A[i][j]))
        A[j], A[p] = A[p], A[j]
        q = 1 / A[j][j]
        A[j] = [v * q for v in A[j]]
        for i in range(n):
            if i != j and A[i][j] != 0:
                t = A[i][j]
                A[i] = [u - t * v for u, v in zip(A[i], A[j])]
    return [r[n:] for r in A]


def _odd_factorial(k):
    return 1 if k <= 0 else k * _odd_factorial(k - 2)


def _signs(a, b):
    return [(a, b), (-a, b), (a, -b), (-a, -b)]


def _basis(d, order):
    """Exponents (e, a, b[, c]) of the basis (p0 - m)^e px^a py^b[ pz^c] up to degree `order` (e <= 1, as
    p0^2 = m^2 + p^2)."""
    out = []
    for e in (0, 1):
        for t in np.ndindex(*([order + 1] * d)):
            if e + sum(t) <= order:
                out.append((e,) + tuple(int(v) for v in t))
    return out


def _weight_moment(e, t, m, d):
    """Mean of (p0 - m)^e p^t under exp(-p0) on the mass shell (m = 0 in three dimensions), as a Decimal."""
    if any(v % 2 for v in t):
        return D(0)
    deg = sum(t)
    ang = D(1)
    for v in t:
        ang *= _odd_factorial(v - 1)
    if d == 3:
        return ang / _odd_factorial(deg + 1) * math.factorial(e + deg + 1)
    for v in range(2, deg + 1, 2):
        ang /= v
    k, rad = deg // 2, D(0)
    for j in range(k + 1):      # (p0 - m)^e ((p0 - m) (2 m + (p0 - m)))^k
        rad += math.comb(k, j) * ((2 * D(m)) ** (k - j) if j < k else 1) * math.factorial(e + k + j)
    return ang * rad


class _Gas:
    """A velocity set in the library's population order with its equilibrium matrix: f^eq = H M(n, U, T)."""

    def __init__(self, d, m, order):
        with decimal.localcontext() as ctx:
            ctx.prec = 60
            self.d, self.m, self.basis = d, float(m), _basis(d, order)
            vec, p, w = {2: self._flat, 3: self._box}[d](m, order)
            G = [[_weight_moment(u[0] + v[0], tuple(x + y for x, y in zip(u[1:], v[1:])), m, d) for v in self.basis]
                 for u in self.basis]
            phi = []
            for q in p:
                row = []
                for u in self.basis:
                    v = (q[0] - D(m)) ** u[0] if u[0] else D(1)
                    for x, a in zip(q[1:], u[1:]):
                        v *= x ** a if a else 1
                    row.append(v)
                phi.append(row)
            X = _solve(G, [list(col) for col in zip(*phi)])           # G^-1 phi^T
            H = [[w[i] * X[k][i] for k in range(len(self.basis))] for i in range(len(p))]
            on = dict(device="cuda", dtype=torch.float64)
            self.n = np.array(vec)
            self.p = torch.tensor([[float(v) for v in q] for q in p], **on)
            self.v = torch.tensor([[float(v / q[0]) for v in q[1:]] for q in p], **on)
            self.H = torch.tensor([[float(v) for v in r] for r in H], **on)
        self.Q = len(vec)

    @staticmethod
    def _flat(m, order):
        if m == 0.0:
            shells, eight, four = {
                2: (["0.4157745567834790", "2.2942803602790417", "6.2899450829374791"],
                    ["0.0888866262411466", "0.0348147166961551", "0.0004218743543938"], ["0", "0", "0.0017535654166088"]),
                3: (["0.3225476896193923", "1.7457611011583465", "4.5366202969211279", "9.3950709123011331"],
                    ["0.0753942630427042", "0.0241670278669858", "0.0026380943565871", "0.0000365655303385"],
                    ["0", "0.0410206173754781", "0.0044457884155769", "0.0000616926157132"])}[order]
            sets = [(s, w, _signs(3, 4) + _signs(4, 3)) for s, w in zip(shells, eight)]
            sets += [(s, w, [(5, 0), (-5, 0), (0, 5), (0, -5)]) for s, w in zip(shells, four) if w != "0"]
            vec = [v for _, _, vs in sets for v in vs]
            # the library holds the tables as doubles: the same numbers here
            p = [(D(float(s)), D(float(s)) * v[0] / 5, D(float(s)) * v[1] / 5) for s, _, vs in sets for v in vs]
            return vec, p, [D(float(w)) for _, w, vs in sets for _ in vs]
        groups, v0 = STENCILS[(m, order)]
        mm, v0 = D(m), D(v0)

        def orbit(g):
            a, b = g
            if b == 0 and a == 0:
                return [(0, 0)]
            if b == 0:
                return [(a, 0), (-a, 0), (0, a), (0, -a)]
            return _signs(a, a) if a == b else _signs(a, b) + _signs(b, a)

        def shell(v):
            g = 1 / (1 - v0 * v0 * (v[0] * v[0] + v[1] * v[1])).sqrt()
            return mm * g, mm * g * v0 * v[0], mm * g * v0 * v[1]

        # weights: moments s^j (j <= 2 N) and |p|^4 cos(4 phi) s^j (j <= 2 N - 4), s = p0 - m
        A, b = [], []
        for j in range(2 * order + 1):
            A.append([sum(((shell(v)[0] - mm) ** j if j else D(1)) for v in orbit(g)) for g in groups])
            b.append([D(math.factorial(j))])
        for j in range(2 * order - 3):
            A.append([sum((x ** 4 - 6 * x * x * y * y + y ** 4) * ((e - mm) ** j if j else 1)
                          for e, x, y in (shell(v) for v in orbit(g))) for g in groups])
            b.append([D(0)])
        w = [r[0] for r in _solve(A, b)]
        kind = [3 if g == (0, 0) else 1 if g[1] == 0 else 2 if g[0] == g[1] else 0 for g in groups]
        sets = [(w[i], orbit(g)) for t in range(4) for i, g in enumerate(groups) if kind[i] == t]
        vec = [v for _, vs in sets for v in vs]
        return vec, [shell(v) for v in vec], [x for x, vs in sets for _ in vs]

    @staticmethod
    def _box(m, order):
        gens, shells, weights = {
            2: ([(2, 2, 1), (3, 0, 0)], ["0.9358222275240878", "3.3054072893322786", "7.7587704831436335"],
                ["0.0245283950433191", "0", "0.0163006691342629", "0", "0.0003891858228425", "0.0017936666649682"]),
            3: ([(4, 4, 3), (5, 4, 0), (6, 2, 1)],
                ["0.7432919279814314", "2.5716350076462784", "5.7311787516890996", "10.953894312683190"],
                ["0", "0", "0.0093098040253911", "0.0085195569675087", "0", "0.0056909667738262", "0.0013041770173120",
                 "0", "0.0008932820065742", "0.0000029126213348", "0.0000338363537565", "0.0000090390475856"])}[order]
        vec, p, w = [], [], []
        for j, s in enumerate(shells):
            for g, gen in enumerate(gens):
                wt = weights[len(gens) * j + g]
                if wt == "0":
                    continue
                orbit = {tuple(s * x for s, x in zip(sign, perm)) for perm in itertools.permutations(gen)
                         for sign in itertools.product((1, -1), repeat=3)}
                length = D(sum(x * x for x in gen)).sqrt()
                for v in sorted(orbit):
                    vec.append(v)
                    p.append((D(float(s)),) + tuple(D(float(s)) * x / length for x in v))
                    w.append(D(float(wt)))
        return vec, p, w

    def moments_of(self, n, U, T):
        """Maxwell-Juettner moments of the basis (App. B), stacked."""
        m, d = self.m, self.d
        if d == 2:
            r0, r2 = 1 / (m + T), (m * m + 3 * m * T + 3 * T * T) / (m + T)
            r3 = (m ** 3 + 6 * m * m * T + 15 * m * T * T + 15 * T ** 3) / (m + T)
        else:
            r0, r2, r3 = 1 / (2 * T), 4 * T, 24 * T * T
        eta = lambda a, b: 0.0 if a != b else 1.0 if a == 0 else -1.0  # noqa: E731

        def raw(idx):
            if len(idx) == 0:
                return n * r0
            if len(idx) == 1:
                return n * U[idx[0]]
            if len(idx) == 2:
                return n * (r2 * U[idx[0]] * U[idx[1]] - T * eta(*idx))
            a, b, c = idx
            return n * (r3 * U[a] * U[b] * U[c] - T * r2 * (eta(a, b) * U[c] + eta(a, c) * U[b] + eta(b, c) * U[a]))

        out = []
        for u in self.basis:
            space = [k + 1 for k, a in enumerate(u[1:]) for _ in range(a)]
            out.append(raw([0] + space) - m * raw(space) if u[0] else raw(space))
        return torch.stack(out)

    def feq(self, n, U, T):
        M = self.moments_of(n, U, T)
        return torch.matmul(self.H, M.reshape(M.shape[0], -1)).reshape((self.Q,) + tuple(n.shape))

    def landau(self, f):
        """n, U, T, eps, N, T^ab of the streamed populations: eps = T00 - t.u and (Tij + eps) u = t, by Newton."""
        d, P = self.d, self.p
        N = torch.tensordot(P.T, f, dims=1)
        Tab = {(a, b): torch.tensordot(P[:, a] * P[:, b], f, dims=1) for a in range(d + 1) for b in range(a, d + 1)}
        lam = Tab[0, 0].detach()
        for it in range(9):
            if it < 7:
                with torch.no_grad():
                    lam, u = self._newton(Tab, lam)
            else:
                lam, u = self._newton(Tab, lam)
        _, u = self._newton(Tab, lam)
        U0 = 1 / torch.sqrt(1 - sum(x * x for x in u))
        U = [U0] + [U0 * x for x in u]
        n = U[0] * N[0] - sum(U[a] * N[a] for a in range(1, d + 1))
        e, m = lam / n, self.m
        if d == 3 or m == 0.0:
            T = e / d
        else:
            T = 0.25 * ((e - 2 * m) + torch.sqrt(e * e + 4 * m * (e - m)))
        return n, U, T, lam, N, Tab

    def _newton(self, Tab, lam):
        d = self.d
        t = [Tab[0, a] for a in range(1, d + 1)]
        if d == 2:
            b, c, r = Tab[1, 1] + lam, Tab[2, 2] + lam, Tab[1, 2]
            D2 = b * c - r * r
            u = [(t[0] * c - r * t[1]) / D2, (t[1] * b - r * t[0]) / D2]
        else:
            a = [[Tab[min(i, j), max(i, j)] + (lam if i == j else 0) for j in (1, 2, 3)] for i in (1, 2, 3)]
            co = [[a[(i + 1) % 3][(j + 1) % 3] * a[(i + 2) % 3][(j + 2) % 3]
                   - a[(i + 1) % 3][(j + 2) % 3] * a[(i + 2) % 3][(j + 1) % 3] for j in range(3)] for i in range(3)]
            D3 = sum(a[0][j] * co[0][j] for j in range(3))
            u = [sum(co[i][j] * t[j] for j in range(3)) / D3 for i in range(3)]
        g = Tab[0, 0] - sum(x * y for x, y in zip(t, u)) - lam
        return lam + g / (1 - sum(x * x for x in u)), u


def _shift(a, sx, sy, clamp):
    """a(x - sx, y - sy): periodic, or in x clamped to the ends."""
    if sy:
        a = torch.roll(a, sy, 0)
    if not clamp:
        return torch.roll(a, sx, 1) if sx else a
    x = (torch.arange(a.shape[1], device=a.device) - sx).clamp(0, a.shape[1] - 1)
    return a[:, x] if sx else a


def _pull(gas, fs, stream, clamp):
    if gas.d == 3:
        return torch.stack([torch.roll(fs[i], tuple(int(s) for s in reversed(gas.n[i])), (0, 1, 2))
                            for i in range(gas.Q)])
    out = []
    for i in range(gas.Q):
        if stream == "onlattice":
            out.append(_shift(fs[i], int(gas.n[i][0]), int(gas.n[i][1]), clamp))
            continue
        src = [-LAM * float(x) for x in gas.v[i]]
        o = [math.floor(s) for s in src]
        px, py = src[0] - o[0], src[1] - o[1]
        out.append(sum(wt * _shift(fs[i], -(o[0] + a), -(o[1] + b), clamp)
                       for a, b, wt in ((0, 0, (1 - px) * (1 - py)), (1, 0, px * (1 - py)), (0, 1, (1 - px) * py),
                                        (1, 1, px * py))))
    return torch.stack(out)


def _collide(gas, f, tau, g=None, walls=False):
    """f* and the fields of f; tau a number, a tensor or a function of T."""
    n, U, T, eps, N, Tab = gas.landau(f)
    feq = gas.feq(n, U, T)
    t = tau(T) if callable(tau) else tau
    vU = torch.tensordot(gas.v, torch.stack(U[1:]), dims=1)
    new = f + (U[0] - vU) / t * (feq - f)
    if g is not None:
        gv = (gas.v @ torch.tensor(g, device="cuda", dtype=torch.float64)).reshape((-1,) + (1,) * n.dim())
        new = new + gas.m / T * feq * (U[0] * gv - sum(x * u for x, u in zip(g, U[1:])))
    if walls:
        one = torch.ones_like(n)
        rest = gas.feq(n, [one] + [0 * one] * gas.d, T)
        new[..., 0], new[..., -1] = rest[..., 0], rest[..., -1]
    return new, (n, U, T, eps, N, Tab)


def _start(gas, f):
    n, *u, T = f
    U0 = 1 / torch.sqrt(1 - sum(x * x for x in u))
    return gas.feq(n, [U0] + [U0 * x for x in u], T)


def _exact_flow(c, seed):
    gas = _Gas(2, c["m"], c["order"])
    fs = _start(gas, _fields2(c["flow"], c["nx"], c["ny"], seed, _T0(c)))
    tau = (lambda T: ETA_S * 4 * KAPPA / T) if c["flow"] == "tube" else c["tau"]
    channel = c["flow"] == "channel"
    for _ in range(c["steps"]):
        f = _pull(gas, fs, c["stream"], c["flow"] in ("tube", "channel"))
        fs, (n, U, T, eps, N, Tab) = _collide(gas, f, tau, GRAVITY if channel else None, channel)
    if c["precision"] == "fp32":
        one = torch.ones(1, device="cuda", dtype=torch.float64)
        fs = fs - gas.feq(one, [one, 0 * one, 0 * one], _T0(c) * one)[:, :, None]
    out = {"n": n, "ux": U[1] / U[0], "uy": None if c["flow"] == "tube" else U[2] / U[0], "T": T, "eps": eps, "N": N,
           "Tab": torch.stack([Tab[k] for k in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))])}
    return {"fields": out, "f": fs}


def _exact_batch(c, seed):
    out, gases = [], {m: _Gas(2, m, 2) for m in (0.0, 1.0, 10.0)}
    for i, (side, tau, m) in enumerate(_sweep(c, seed)):
        gas = gases[m]
        fs = _start(gas, _fields2("shear", side, side, seed + i))
        for _ in range(c["steps"]):
            fs, _f = _collide(gas, _pull(gas, fs, "onlattice", False), tau)
        one = torch.ones(1, device="cuda", dtype=torch.float64)
        out.append(fs - gas.feq(one, [one, 0 * one, 0 * one], one)[:, :, None])
    return out


def _exact_flow3(c, seed):
    gas = _Gas(3, 0.0, c["order"])
    if gas.Q * c["nx"] * c["ny"] * c["nz"] > 6e8:
        return None
    fs = _start(gas, _fields3(c["nx"], c["ny"], c["nz"], seed))
    for _ in range(c["steps"]):
        f = _pull(gas, fs, "onlattice", False)
        fs, (n, U, T, eps, _N, _Tab) = _collide(gas, f, c["tau"])
    return {"n": n, "ux": U[1] / U[0], "uy": U[2] / U[0], "uz": U[3] / U[0], "T": T, "eps": eps}


def _exact_wave(c, seed):
    """(1+1) dimensions: the 2 N populations p0_j (1, +-1) carry the moments n (a-1)! T^(a-1) {cosh, sinh}(a theta) of
    the members p0^a and p0^a sign(px), a = 1..N, of the equilibrium."""
    N = c["order"]
    x = {2: ["3.414213562373095048", "0.585786437626904951"],
         3: ["6.289945082937479196", "0.415774556783479083", "2.294280360279041719"],
         4: ["0.322547689619392311", "4.536620296921127983", "9.395070912301133129", "1.745761101158346575"],
         5: ["0.26356031971814091020", "3.59642577104072208122", "1.41340305910651679221", "7.08581000585883755692",
             "12.6408008442757826594"]}[N]
    with decimal.localcontext() as ctx:
        ctx.prec = 60
        pops = [(D(float(v)), s) for v in x for s in (1, -1)]
        A = [[p ** a * (s if b else 1) for p, s in pops] for a in range(1, N + 1) for b in (0, 1)]
        inv = _solve(A, [[D(int(i == j)) for j in range(2 * N)] for i in range(2 * N)])
        H = torch.tensor([[float(v) for v in r] for r in inv], device="cuda", dtype=torch.float64)
    p0 = torch.tensor([float(p) for p, _ in pops], device="cuda", dtype=torch.float64)[:, None]
    sg = torch.tensor([float(s) for _, s in pops], device="cuda", dtype=torch.float64)[:, None]

    def feq(n, U0, Ux, T):
        M = []
        for a in range(1, N + 1):
            k = 0.5 * n * math.factorial(a - 1) * T ** (a - 1)
            M += [k * ((U0 + Ux) ** a + (U0 + Ux) ** -a), k * ((U0 + Ux) ** a - (U0 + Ux) ** -a)]
        return torch.matmul(H, torch.stack(M))

    n, u, T = _fields1(c["nx"], seed)
    U0 = 1 / torch.sqrt(1 - u * u)
    fs = feq(n, U0, U0 * u, T)
    for _ in range(c["steps"]):
        f = torch.stack([torch.roll(fs[i], s, 0) for i, (_, s) in enumerate(pops)])
        N0, Nx, E, F = (f * p0).sum(0), (f * p0 * sg).sum(0), (f * p0 * p0).sum(0), (f * p0 * p0 * sg).sum(0)
        eps = torch.sqrt((E - F) * (E + F))
        u = F / (E + eps)
        U0 = 1 / torch.sqrt(1 - u * u)
        n = U0 * (N0 - u * Nx)
        T = eps / n
        fs = f + U0 * (1 - sg * u) / c["tau"] * (feq(n, U0, U0 * u, T) - f)
    return dict(zip([name for name, _ in PLANES1], (n, u, T, eps, N0, Nx, E, F)))


def _exact_adjoint(c, seed):
    if c["steps"] * c["nx"] * c["ny"] > 2.6e7:
        return None
    gas = _Gas(2, 0.0, 2)
    n, ux, uy, T = _fields2("shear", c["nx"], c["ny"], seed)
    target = _target(c, (n, ux, uy, T))
    ux, uy = ux.requires_grad_(), uy.requires_grad_()
    tau = torch.ones_like(n, requires_grad=True)
    states = [_start(gas, (n, ux, uy, T))]
    # states without a graph first, then back through them step by step
    with torch.no_grad():
        x = states[0].detach()
        xs = [x]
        for _ in range(c["steps"]):
            x, _f = _collide(gas, _pull(gas, x, c["stream"], False), tau)
            xs.append(x)
    last = xs[c["steps"] - 1].detach().requires_grad_()
    _n, U, *_r = gas.landau(_pull(gas, last, c["stream"], False))
    loss = 0.5 * ((U[1] / U[0] - target[0]) ** 2 + (U[2] / U[0] - target[1]) ** 2).sum()
    (a,) = torch.autograd.grad(loss, last)
    g_tau = torch.zeros_like(n)
    for k in range(c["steps"] - 1, 0, -1):
        x = xs[k - 1].detach().requires_grad_()
        y, _f = _collide(gas, _pull(gas, x, c["stream"], False), tau)
        a, gt = torch.autograd.grad(y, (x, tau), a)
        g_tau += gt
    g_ux, g_uy = torch.autograd.grad(states[0], (ux, uy), a)
    return {"tau": g_tau, "ux0": g_ux, "uy0": g_uy}


def exact(case, seed):
    """What a pass on a new state returns, in 64 bits; None where that would take too long."""
    return {"flow": _exact_flow, "batch": _exact_batch, "flow3": _exact_flow3, "wave": _exact_wave,
            "adjoint": _exact_adjoint}[case["kind"]](case, seed)
