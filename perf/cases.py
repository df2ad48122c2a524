"""Timed cases of the solver: what a program using this package has it do,
through the public entry points of ``paper_1206_1361_gb300.gp``.

A case is one of three kinds of work:

* ``grid``: one context (``gp.Solver``): load a state that is on the GPU,
  take some SSCN steps, read the observables, store the state -- one report
  interval of a single-grid run.  Three precisions, imaginary and real time,
  2D and 3D, the plain and the symmetric splitting, constant and modulated g.
* ``axial``: the same on the axially symmetric form (``gp.Solver.axial``).
* ``batch``: many resident problems (``gp.Batch``) advanced together by some
  steps, then the observables and the states of all of them -- one turn of
  the serving loop.

``exact`` is the same method in plain torch FP64: each Crank-Nicolson sweep as
a dense matrix (I - kappa L)^-1 (I + kappa L) applied along its axis.
"""
import math

import numpy as np
import torch

from paper_1206_1361_gb300 import gp, workloads

PRECISIONS = {"c128": gp.GP_C128, "c64": gp.GP_C64, "ff": gp.GP_CFF}
POINT_BYTES = {"c128": 16, "c64": 8, "ff": 16}
OBSERVABLES = ("norm", "mu", "energy", "rms_x", "rms_y", "rms_z", "rms_r")


def _grid(name, shape, h, dt, trap, g, mode, precision, steps, strang=False, g1=0.0, omega=0.0):
    case = {"kind": "grid", "nx": shape[0], "ny": shape[1], "nz": shape[2],
            "hx": h[0], "hy": h[1], "hz": h[2], "dt": dt,
            "wx": trap[0], "wy": trap[1], "wz": trap[2], "g": g, "real": bool(mode),
            "precision": precision, "steps": steps, "strang": strang, "g1": g1, "omega": omega}
    if name:
        case["name"] = name
    return case


def _recipe(name, shape, trap, g, mode, precision, steps, kappa=0.05, **more):
    """A grid of the batched and served problems: the box spans six radii a
    side; kappa = dt / (4 min h^2) is 0.05 for their dt = 0.2 min h^2."""
    h, dt = workloads.box_spacing(shape, trap, g)
    return _grid(name, shape, h, dt * kappa / 0.05, trap, g, mode, precision, steps, **more)


def listed():
    small, quench, large = (workloads.SMALL_IMAG_64, workloads.REAL_256, workloads.PRECISION_512)
    every = quench.extra["report_every"]
    return [
        # the smallest calls: a small ground-state solve checked every 10 steps
        _recipe("check-48x32x32-c128", (48, 32, 32), (1.0, 1.5, 2.0), 40.0, 0, "c128", 10),
        # the small ground-state run: 64^3, the default precision
        _grid("ground-64-c128", small.shape, small.h, small.dt, small.trap, small.g, 0, "c128", 100),
        # 2D ground state, uneven edges
        _recipe("ground-2d-500x384-c128", (500, 384, 1), (1.0, 1.7, 0.0), 120.0, 0, "c128", 40),
        # real-time run with a modulated interaction and the symmetric splitting
        _recipe("faraday-128x96x80-c128", (128, 96, 80), (1.0, 1.5, 2.0), 60.0, 1, "c128", 20,
                strang=True, g1=20.0, omega=6.0),
        # ground state on a grid of odd edges, single precision
        _recipe("ground-193x130x97-c64", (193, 130, 97), (0.8, 1.3, 2.2), 150.0, 0, "c64", 20),
        # one report interval of the 256^3 quench: FP64-class pairs, and FP64
        _grid("quench-256-ff", quench.shape, quench.h, quench.dt, quench.trap, quench.g, 1, "ff", every),
        _grid("quench-256-c128", quench.shape, quench.h, quench.dt, quench.trap, quench.g, 1, "c128", every),
        # the large single-precision run
        _grid("large-512x512x256-c64", large.shape, large.h, large.dt, large.trap, large.g, 1, "c64", 10),
        # axially symmetric dynamics
        {"name": "axial-1024x2048", "kind": "axial", "nr": 1024, "nz": 2048, "hr": 0.0125, "hz": 0.0125,
         "dt": 1e-5, "wr": 1.0, "wz": 4.0, "g": 100.0, "real": True, "steps": 10},
        # 256 small ground-state solves at once; a mix of served ground states
        # and quenches; the last solve of a batch, alone
        {"name": "batch-256", "kind": "batch", "set": "batched", "count": 256, "offset": 0, "steps": 16},
        {"name": "serve-60", "kind": "batch", "set": "requests", "count": 60, "offset": 0, "steps": 10},
        {"name": "last-of-batch", "kind": "batch", "set": "lone", "count": 1, "offset": 0, "steps": 50},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["grid"] * 5 + ["axial"] + ["batch"] * 2)
    if kind == "batch":
        which = rng.choice(["batched", "requests"])
        count = log(1, 256) if which == "batched" else log(1, 60)
        return {"kind": "batch", "set": which, "count": count, "offset": rng.randrange(0, 257 - count),
                "steps": rng.choice([8, 10, 16])}
    real = rng.random() < 0.5
    if kind == "axial":
        nr, nz = log(48, 1024), log(64, 2048)
        hr, hz = 12.0 / nr, 20.0 / nz
        return {"kind": "axial", "nr": nr, "nz": nz, "hr": hr, "hz": hz,
                "dt": rng.uniform(0.01, 0.2) * min(hr, hz) ** 2, "wr": 1.0, "wz": rng.uniform(0.5, 4.0),
                "g": rng.uniform(0.0, 200.0), "real": real, "steps": rng.choice([10, 20])}
    precision = rng.choice(["c128", "c128", "c64", "ff"])
    most = 2 ** 26 if precision == "c64" else 2 ** 24
    if rng.random() < 0.25:
        shape = (log(64, 2048), log(64, 2048), 1)
    else:
        shape = (log(24, 512), log(24, 512), log(24, 512))
        while shape[0] * shape[1] * shape[2] > most:
            shape = tuple(max(24, int(0.9 * n)) for n in shape)
    if rng.random() < 0.5:                 # half of the grids have rows of 16 or 32 bytes
        shape = (shape[0] + (-shape[0]) % 4,) + shape[1:]
        while shape[0] * shape[1] * shape[2] > most:
            shape = (shape[0] - 4,) + shape[1:]
    trap = tuple(rng.uniform(0.5, 4.0) for _ in range(3))
    if shape[2] == 1:
        trap = trap[:2] + (0.0,)
    kappa = math.exp(rng.uniform(math.log(0.004), math.log(0.018 if precision == "ff" else 0.05)))
    strang = precision != "ff" and rng.random() < 0.2
    g = rng.uniform(0.0, 200.0)
    modulated = rng.random() < 0.15
    steps = max(5, min(100, 10 * round(2 ** 24 / (shape[0] * shape[1] * shape[2]))))
    return _recipe(None, shape, trap, g, int(real), precision, steps, kappa=kappa, strang=strang,
                   g1=0.3 * g if modulated else 0.0, omega=6.0 if modulated else 0.0)


# ------------------------------------------------------------------- inputs

def _axis(n, h):
    return (torch.arange(n, dtype=torch.float64, device="cuda") - 0.5 * n) * h if n > 1 else \
        torch.zeros(1, dtype=torch.float64, device="cuda")


def _uniform(rng, lo, hi):
    return float(rng.uniform(lo, hi))


def _factor(rng, x, half, real):
    """One axis of a condensate-like state: a displaced Gaussian of a third of
    the box's half width, with a long-wave ripple and (real time) a slow phase."""
    w = half * _uniform(rng, 0.25, 0.4)
    u = (x - half * _uniform(rng, -0.1, 0.1)) / w
    f = torch.exp(-0.5 * u * u) * (1.0 + 0.1 * torch.cos(_uniform(rng, 1.0, 3.0) * u + _uniform(rng, 0.0, 6.0)))
    return f * torch.exp(1j * _uniform(rng, 0.2, 1.5) * u) if real else f.to(torch.complex128)


def _noise(seed, shape, envelope):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    re = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)
    im = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)
    return torch.complex(re, im) * envelope


def _cartesian_state(shape, h, real, seed, dtype):
    """A normalised state (nz, ny, nx), zero on the Dirichlet nodes: two
    overlapping condensate-like lumps and a little noise where they are."""
    rng = np.random.Generator(np.random.PCG64(seed))
    axes = [(_axis(n, hk), 0.5 * n * hk) for n, hk in zip(shape, h)]
    psi = None
    for amplitude in (1.0, 0.3):
        fx, fy, fz = (_factor(rng, x, half, real) if len(x) > 1 else torch.ones_like(x, dtype=torch.complex128)
                      for x, half in axes)
        term = amplitude * fz[:, None, None] * fy[None, :, None] * fx[None, None, :]
        psi = term if psi is None else psi + term
    if real:
        psi += 1e-3 * _noise(seed, psi.shape, psi.abs())
    psi[:, 0, :] = 0
    psi[:, :, 0] = 0
    if shape[2] > 1:
        psi[0] = 0
    w = h[0] * h[1] * (h[2] if shape[2] > 1 else 1.0)
    psi /= torch.sqrt(w * psi.abs().square().sum())
    return psi.to(dtype)


def _axial_state(c, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    rho = (torch.arange(c["nr"], dtype=torch.float64, device="cuda") + 0.5) * c["hr"]
    z = _axis(c["nz"], c["hz"])
    a = _uniform(rng, 0.2, 0.35) * c["nr"] * c["hr"]
    fr = torch.exp(-0.5 * (rho / a) ** 2) * (1.0 + 0.1 * torch.cos(_uniform(rng, 1.0, 3.0) * (rho / a) ** 2))
    psi = _factor(rng, z, 0.5 * c["nz"] * c["hz"], c["real"])[:, None] * fr[None, :]
    if c["real"]:
        psi = psi + 1e-3 * _noise(seed, psi.shape, psi.abs())
    psi[0] = 0
    w = 2.0 * math.pi * c["hr"] * c["hz"]
    return psi / torch.sqrt(w * (rho[None, :] * psi.abs().square()).sum())


def _batch_set(case):
    """(instance, mode, g of the step) of the problems resident in the batch."""
    if case["set"] == "lone":
        shape, trap, g = (128, 128, 32), (0.9, 1.1, 3.5), 150.0
        h, dt = workloads.box_spacing(shape, trap, g)
        return [(workloads.Instance(shape, h, dt, trap, g), gp.GP_IMAG, g)]
    a, b = case["offset"], case["offset"] + case["count"]
    if case["set"] == "batched":
        return [(i, gp.GP_IMAG, i.g) for i in workloads.batched_instances()[a:b]]
    return [(r.inst, gp.GP_REAL, r.quench_g) if r.kind == "quench" else (r.inst, gp.GP_IMAG, r.inst.g)
            for r in workloads.request_stream(count=b)[a:b]]


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        # the states stay in the batch, as between two turns of a serving loop
        problems = _batch_set(c)
        batch = gp.Batch(gp.GP_C64, cap_bytes=1 << 35)
        total = sum(i.points for i, _, _ in problems)
        out = torch.empty(total, dtype=torch.complex64, device="cuda")
        slots, at = [], 0
        for k, (i, mode, g) in enumerate(problems):
            psi = _cartesian_state(i.shape, i.h, mode == gp.GP_REAL, seed * 1000 + k, torch.complex64)
            torch.cuda.synchronize()
            slot = batch.add(i.shape, i.h, i.dt, *i.trap, g, mode, psi=psi)
            slots.append((slot, out[at:at + i.points]))
            at += i.points
        return {"kind": "batch", "batch": batch, "slots": slots, "out": out, "steps": c["steps"]}
    if c["kind"] == "axial":
        psi = _axial_state(c, seed)
        solver = gp.Solver.axial(c["nr"], c["nz"], c["hr"], c["hz"], c["dt"], c["wr"], c["wz"], c["g"],
                                 gp.GP_REAL if c["real"] else gp.GP_IMAG)
    else:
        shape, h = (c["nx"], c["ny"], c["nz"]), (c["hx"], c["hy"], c["hz"])
        dtype = torch.complex64 if c["precision"] == "c64" else torch.complex128
        psi = _cartesian_state(shape, h, c["real"], seed, dtype)
        solver = gp.Solver(shape, h, c["dt"], c["wx"], c["wy"], c["wz"], c["g"],
                           gp.GP_REAL if c["real"] else gp.GP_IMAG, PRECISIONS[c["precision"]])
        if c["strang"]:
            solver.set_splitting(gp.GP_SPLIT_STRANG)
        if c["g1"]:
            solver.set_modulation(c["g1"], c["omega"])
    torch.cuda.synchronize()
    return {"kind": c["kind"], "solver": solver, "psi": psi, "out": torch.empty_like(psi), "steps": c["steps"]}


def run(state):
    if state["kind"] == "batch":
        batch = state["batch"]
        batch.step(state["steps"])
        seen = batch.observables()
        for slot, part in state["slots"]:
            gp.gp_batch_store(batch.b, slot, part)
        return {"psi": state["out"],
                "obs": np.array([[seen[slot][k] for k in OBSERVABLES] for slot, _ in state["slots"]])}
    solver = state["solver"]
    solver.load(state["psi"])
    solver.step(state["steps"])
    seen = solver.observables()
    gp.gp_store(solver.ctx, state["out"])
    return {"psi": state["out"], "obs": np.array([seen[k] for k in OBSERVABLES]), "step": seen["step"]}


def work(case):
    """Each step reads the state and writes it once, a report reads it once;
    operations as the method's formulas count them (a complex multiply 6, an
    exponential or a sine-cosine pair 1)."""
    def one(points, axes, real, e, steps, strang=False):
        step = axes * (28 if real else 18) + (13 if real else 11) * (2 if strang else 1)
        return points * e * (2 * steps + 1), points * (step * steps + 30)

    if case["kind"] == "batch":
        parts = [one(i.points, 3 if i.shape[2] > 1 else 2, mode == gp.GP_REAL, 8, case["steps"])
                 for i, mode, _ in _batch_set(case)]
    elif case["kind"] == "axial":
        parts = [one(case["nr"] * case["nz"], 2, case["real"], 16, case["steps"])]
    else:
        parts = [one(case["nx"] * case["ny"] * case["nz"], 3 if case["nz"] > 1 else 2, case["real"],
                     POINT_BYTES[case["precision"]], case["steps"], case["strang"])]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


# -------------------------------------------------------------- 64-bit truth

def _tridiag(lower, upper):
    return torch.diag(torch.full((len(lower) + 1,), -2.0, dtype=torch.float64)) + \
        torch.diag(lower, -1) + torch.diag(upper, 1)


def _sweep_matrix(lap, h, dt, real):
    """(I - kappa L)^-1 (I + kappa L), kappa = dt / (4 h^2) (times i in real time)."""
    k = dt / (4.0 * h * h)
    eye = torch.eye(len(lap), dtype=torch.float64)
    if real:
        return torch.linalg.solve(torch.complex(eye, -k * lap), torch.complex(eye, k * lap)).cuda()
    return torch.linalg.solve(eye - k * lap, eye + k * lap).cuda()


def _apply(matrix, psi, dim):
    """matrix along dim of psi, a slab of the other axes at a time."""
    moved = psi.movedim(dim, 0)
    flat = moved.reshape(moved.shape[0], -1)
    out = torch.empty_like(flat)
    for a in range(0, flat.shape[1], 1 << 19):
        part = flat[:, a:a + (1 << 19)]
        if matrix.is_complex():
            out[:, a:a + (1 << 19)] = matrix @ part
        else:
            out[:, a:a + (1 << 19)] = torch.complex(matrix @ part.real, matrix @ part.imag)
    return out.reshape(moved.shape).movedim(0, dim)


class _Truth:
    """The method on one grid in FP64: axes in storage order (slowest first)."""

    def __init__(self, sweeps, potential, volume, weight, g, dt, real, strang=False, g1=0.0, omega=0.0):
        self.sweeps, self.v, self.volume, self.weight = sweeps, potential, volume, weight
        self.g, self.dt, self.real, self.strang, self.g1, self.omega = g, dt, real, strang, g1, omega
        self.step = 0

    def big_g(self, fa, fb):
        ta, tb = (self.step + fa) * self.dt, (self.step + fb) * self.dt
        if not self.g1:
            return self.g * (tb - ta)
        return self.g * (tb - ta) + self.g1 * (math.sin(self.omega * tb) - math.sin(self.omega * ta)) / self.omega

    def pointwise(self, psi, fa, fb):
        a = self.v * ((fb - fa) * self.dt) + self.big_g(fa, fb) * psi.abs().square()
        return psi * (torch.exp(-1j * a) if self.real else torch.exp(-a))

    def normalised(self, psi):
        return psi if self.real else psi / torch.sqrt(self.volume * (self.weight * psi.abs().square()).sum())

    def advance(self, psi, steps):
        for _ in range(steps):
            psi = self.pointwise(psi, 0.0, 0.5 if self.strang else 1.0)
            for matrix, dim in self.sweeps:
                inner = psi.narrow(dim, psi.shape[dim] - len(matrix), len(matrix))
                psi = psi.clone()
                psi.narrow(dim, psi.shape[dim] - len(matrix), len(matrix)).copy_(_apply(matrix, inner, dim))
            psi = self.normalised(psi)
            if self.strang:
                psi = self.normalised(self.pointwise(psi, 0.5, 1.0))
            self.step += 1
        return psi

    def g_now(self):
        return self.g + self.g1 * math.cos(self.omega * self.step * self.dt)


def _differences(psi, dim):
    """Squared forward differences along dim; the node past the end is zero."""
    end = torch.zeros_like(psi.narrow(dim, 0, 1))
    return torch.diff(torch.cat([psi, end], dim), dim=dim).abs().square()


def _cartesian_truth(shape, h, dt, trap, g, real, psi, steps, **more):
    nd = 3 if shape[2] > 1 else 2
    sweeps, potential, squares = [], 0.0, []
    for k in range(3):
        dim = 2 - k                        # x is the fastest axis of (nz, ny, nx)
        x2 = (_axis(shape[k], h[k]) ** 2).reshape([-1 if d == dim else 1 for d in range(3)])
        squares.append(x2)
        potential = potential + 0.5 * trap[k] ** 2 * x2
        if k < nd:
            one = torch.ones(shape[k] - 2, dtype=torch.float64)
            sweeps.append((_sweep_matrix(_tridiag(one, one), h[k], dt, real), dim))
    volume = h[0] * h[1] * (h[2] if nd == 3 else 1.0)
    truth = _Truth(sweeps, potential, volume, 1.0, g, dt, real, **more)
    psi = truth.advance(psi, steps)
    a = psi.abs().square()
    s0 = float(a.sum())
    kin = sum(0.5 * float(_differences(psi, 2 - k).sum()) / h[k] ** 2 for k in range(nd))
    pot, quart = float((potential * a).sum()), truth.g_now() * float(a.square().sum())
    moments = [float((x2 * a).sum()) / s0 for x2 in squares]
    obs = [volume * s0, (kin + pot + quart) / s0, (kin + pot + 0.5 * quart) / s0,
           *(math.sqrt(m) for m in moments), math.sqrt(sum(moments))]
    return psi, np.array(obs)


def _axial_truth(c, psi):
    nr, nz, hr, hz = c["nr"], c["nz"], c["hr"], c["hz"]
    i = torch.arange(nr, dtype=torch.float64)
    lap_r = _tridiag((1.0 - 1.0 / (2.0 * i + 1.0))[1:], (1.0 + 1.0 / (2.0 * i + 1.0))[:-1])
    one = torch.ones(nz - 2, dtype=torch.float64)
    sweeps = [(_sweep_matrix(lap_r, hr, c["dt"], c["real"]), 1),
              (_sweep_matrix(_tridiag(one, one), hz, c["dt"], c["real"]), 0)]
    rho = ((i.cuda() + 0.5) * hr)[None, :]
    z = _axis(nz, hz)[:, None]
    potential = 0.5 * (c["wr"] ** 2 * rho ** 2 + c["wz"] ** 2 * z ** 2)
    volume = 2.0 * math.pi * hr * hz
    truth = _Truth(sweeps, potential, volume, rho, c["g"], c["dt"], c["real"])
    psi = truth.advance(psi, c["steps"])
    a = psi.abs().square()
    s0 = float((rho * a).sum())
    kin = 0.5 * float(((rho + 0.5 * hr) * _differences(psi, 1)).sum()) / hr ** 2 + \
        0.5 * float((rho * _differences(psi, 0)).sum()) / hz ** 2
    pot, quart = float((rho * potential * a).sum()), c["g"] * float((rho * a.square()).sum())
    r2, z2 = float((rho ** 3 * a).sum()) / s0, float((rho * z ** 2 * a).sum()) / s0
    obs = [volume * s0, (kin + pot + quart) / s0, (kin + pot + 0.5 * quart) / s0,
           math.sqrt(0.5 * r2), math.sqrt(0.5 * r2), math.sqrt(z2), math.sqrt(r2 + z2)]
    return psi, np.array(obs)


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        psis, rows = [], []
        for k, (i, mode, g) in enumerate(_batch_set(c)):
            psi = _cartesian_state(i.shape, i.h, mode == gp.GP_REAL, seed * 1000 + k, torch.complex64)
            psi, obs = _cartesian_truth(i.shape, i.h, i.dt, i.trap, g, mode == gp.GP_REAL,
                                        psi.to(torch.complex128), c["steps"])
            psis.append(psi.reshape(-1))
            rows.append(obs)
        return {"psi": torch.cat(psis), "obs": np.array(rows)}
    if c["kind"] == "axial":
        psi, obs = _axial_truth(c, _axial_state(c, seed))
    else:
        shape, h = (c["nx"], c["ny"], c["nz"]), (c["hx"], c["hy"], c["hz"])
        dtype = torch.complex64 if c["precision"] == "c64" else torch.complex128
        psi = _cartesian_state(shape, h, c["real"], seed, dtype).to(torch.complex128)
        psi, obs = _cartesian_truth(shape, h, c["dt"], (c["wx"], c["wy"], c["wz"]), c["g"], c["real"], psi,
                                    c["steps"], strang=c["strang"], g1=c["g1"], omega=c["omega"])
    return {"psi": psi, "obs": obs, "step": c["steps"]}
