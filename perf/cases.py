"""What is measured: the calls a user of this library makes, from the
smallest grids to the largest, each through a public entry point.

A case is a dict of plain values.  ``kind`` names the call:

* ``poisson``: one standalone Poisson solve to a tolerance, rhs and solution
  on the device (vsv_solve_poisson);
* ``step``: time steps of one body in a channel (vsv_step), after which the
  program reads phi and the velocity;
* ``batch``: time steps of one or many grids through the captured graph
  (vsv_batch_step);
* ``adjoint``: the gradient of a trajectory (the tape: forward run with
  checkpoints, then the reverse pass);
* ``observe``: the observables of a state (diagnostics, stress profile,
  velocity and in-plane stress fields).

``exact`` evaluates the same discrete problem in 64 bits with torch alone:
Poisson problems by the orthonormal sine / Fourier basis of each axis, steps
by the finite differences they are defined with, gradients by torch.autograd
through those steps.
"""
import math

import numpy as np
import torch

from paper_2601_05031_gb300 import vsv as V
from paper_2601_05031_gb300.adjoint import Tape
from paper_2601_05031_gb300.sim import Batch, Simulation

DUCT, PLANAR, COUETTE = V.VSV_POISEUILLE_DUCT, V.VSV_POISEUILLE_PLANAR, V.VSV_COUETTE
CH, HELFRICH = V.VSV_CAHN_HILLIARD, V.VSV_HELFRICH


def _poisson(name, nx, ny, nz, prec, tol, per_x=1, per_y=0, per_z=0, solver="mg", shift=0.0):
    return {"name": name, "kind": "poisson", "nx": nx, "ny": ny, "nz": nz, "prec": prec, "tol": tol,
            "per_x": per_x, "per_y": per_y, "per_z": per_z, "solver": solver, "shift": shift}


def _step(name, nx, ny, nz, prec, body, flow, steps, cycles=0, order=1, tol=1e-10, solver="mg",
          dt=1e-4, eps=1.0, vr=0.8, rho=0.0, kind="step"):
    return {"name": name, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "prec": prec, "body": body,
            "flow": flow, "steps": steps, "cycles": cycles, "order": order, "tol": tol,
            "solver": solver, "dt": dt, "eps": eps, "vr": vr, "rho": rho}


def listed():
    return [
        # the validation run: a small droplet in a duct, plain FP64, every solve
        # by red-black SOR to 1e-10 (latency: a few thousand cells per kernel)
        _step("droplet_fp64_sor_48x24x24", 48, 24, 24, "fp64", "droplet", DUCT, 10, solver="sor",
              dt=0.01),
        # a small standalone solve, as a coupling code or a test calls it
        _poisson("poisson_mixed_64x32x32", 64, 32, 32, "mixed", 1e-9),
        # a mid-size standalone solve in plain FP64 with every wall present and
        # extents that are no powers of two
        _poisson("poisson_fp64_112x72x56", 112, 72, 56, "fp64", 1e-10, per_x=0),
        # the largest solve: one component at the benchmark's size
        _poisson("poisson_mixed_512x256x256", 512, 256, 256, "mixed", 1e-9, per_z=1),
        # the library's default solver settings (every solve to its tolerance) on
        # a ragged grid, inertial droplet between plates: the shifted operator
        _step("droplet_inertial_default_192x96x80", 192, 96, 80, "mixed", "droplet", PLANAR, 3,
              rho=0.01),
        # parameter-fitting size, plain stepping with the fixed schedule
        _step("vesicle_duct_128x64x64", 128, 64, 64, "mixed", "vesicle", DUCT, 8, cycles=2, order=2),
        # production run of a single vesicle, plain stepping
        _step("vesicle_duct_256x128x128", 256, 128, 128, "mixed", "vesicle", DUCT, 6, cycles=2,
              order=2),
        # the benchmark: one large Couette vesicle through the captured graph
        _step("vesicle_couette_512x256x256", 512, 256, 256, "mixed", "vesicle", COUETTE, 6, cycles=2,
              order=2, eps=1.5, vr=0.9, kind="batch"),
        # the plain FP64 step beside it, at the size where a user still runs it
        _step("vesicle_couette_fp64_256x128x128", 256, 128, 128, "fp64", "vesicle", COUETTE, 2,
              cycles=2, order=2, eps=1.5, vr=0.9),
        # a parameter sweep: many small grids of uneven sizes in one graph
        {"name": "sweep_12_grids", "kind": "batch", "grids": 12, "lo": 32, "hi": 96, "steps": 12,
         "cycles": 2, "order": 2, "dt": 1e-4, "prec": "mixed", "sizes": 5},
        # a gradient for the fit of membrane parameters
        dict(_step("gradient_128x64x64", 128, 64, 64, "mixed", "vesicle", DUCT, 10, cycles=2, order=2,
                   kind="adjoint"), every=5, adj_cycles=4),
        # observables of a state, as a run writes them out every few steps
        _step("observables_256x128x128", 256, 128, 128, "mixed", "vesicle", DUCT, 0, kind="observe"),
    ]


def _log_int(rng, lo, hi, mult):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, int(round(v / mult)) * mult)


def _sizes(rng, lo, hi, mult):
    """(nx, ny, nz): ny, nz log-uniform in lo .. hi, nx up to twice that."""
    ny, nz = _log_int(rng, lo, hi, mult), _log_int(rng, lo, hi, mult)
    return _log_int(rng, lo, 2 * hi, mult), ny, nz


def draw(rng):
    case = _drawn(rng)
    case.pop("name", None)
    return case


def _drawn(rng):
    # sizes are multiples of 16 where solves iterate to a tolerance, so that a
    # multigrid hierarchy exists
    k = rng.choice(["poisson", "poisson", "step", "step", "default", "fp64", "batch", "adjoint",
                    "observe"])
    if k == "poisson":
        prec = rng.choice(["mixed", "mixed", "fp64"])
        nx, ny, nz = _sizes(rng, 32, 256 if prec == "mixed" else 128, 16)
        per_z = rng.randint(0, 1)
        return _poisson(None, nx, ny, nz, prec, 1e-9, per_x=rng.choice([1, 1, 1, 0]),
                        per_y=rng.choice([0, 0, 0, 1]) * (1 - per_z), per_z=per_z,
                        shift=rng.choice([0.0, 0.0, 0.3]))
    if k == "batch":
        return {"kind": "batch", "grids": rng.randint(2, 12), "lo": 32, "hi": rng.choice([48, 64, 96]),
                "steps": 12, "cycles": 2, "order": rng.randint(1, 2), "dt": 1e-4, "prec": "mixed",
                "sizes": rng.randint(1, 10 ** 6)}
    body = rng.choice(["vesicle", "droplet"])
    flow = rng.choice([DUCT, PLANAR, COUETTE])
    vr, eps = round(rng.uniform(0.7, 0.98), 3), rng.choice([1.0, 1.25, 1.5])
    if k == "step":
        nx, ny, nz = _sizes(rng, 32, 192, 16)
        return _step(None, nx, ny, nz, "mixed", body, flow, 6, cycles=rng.randint(2, 3), order=2,
                     eps=eps, vr=vr)
    if k == "default":
        nx, ny, nz = _sizes(rng, 32, 112, 16)
        return _step(None, nx, ny, nz, "mixed", body, flow, 3, eps=eps, vr=vr,
                     rho=rng.choice([0.0, 0.01]))
    if k == "fp64":
        sor = rng.random() < 0.5
        nx, ny, nz = _sizes(rng, 24 if sor else 32, 40 if sor else 112, 4 if sor else 16)
        return _step(None, nx, ny, nz, "fp64", body, flow, 2, cycles=0 if sor else rng.choice([0, 2]),
                     order=1, solver="sor" if sor else "mg", eps=eps, vr=vr)
    nx, ny, nz = _sizes(rng, 32, 96, 16)
    if k == "adjoint":
        return dict(_step(None, nx, ny, nz, "mixed", body, flow, rng.randint(3, 8), cycles=2, order=2,
                          kind="adjoint", eps=eps, vr=vr), every=rng.randint(2, 5), adj_cycles=4)
    return _step(None, nx, ny, nz, "mixed", body, flow, 0, kind="observe", eps=eps, vr=vr)


# ---------------------------------------------------------------- inputs
def _axis(vr):
    """Aspect a / b of the prolate spheroid of reduced volume vr."""
    def red(s):
        if s <= 1.0 + 1e-9:
            return 1.0
        e = math.sqrt(1.0 - 1.0 / (s * s))
        area = 2.0 * math.pi * (1.0 + s / e * math.asin(e))
        return s / (area / (4.0 * math.pi)) ** 1.5
    lo, hi = 1.0, 50.0
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if red(mid) > vr else (lo, mid)
    return 0.5 * (lo + hi)


def _scene(case, seed):
    """phi0 and the physical parameters: a sphere (Cahn-Hilliard droplet) or a
    prolate spheroid along x (Helfrich vesicle) near the channel's centre."""
    rng = np.random.default_rng(seed)
    nx, ny, nz, eps = case["nx"], case["ny"], case["nz"], case["eps"]
    zper = case["flow"] in (PLANAR, COUETTE)
    p = dict(flow=case["flow"], eps=eps, mobility=1.0, zper=zper, rho=case.get("rho", 0.0),
             u_max=0.0, v_lo=0.0, v_hi=0.0, sigma=0.0, kappa=0.0, k_area=0.0, k_vol=0.0,
             dt=case["dt"], nx=nx, ny=ny, nz=nz)
    H = ny + 1.0
    if case["flow"] == COUETTE:
        p.update(v_lo=-0.05, v_hi=0.05)
        shear = 0.1 / H
    else:
        p.update(u_max=0.05)
        shear = 0.2 / H
    if case["body"] == "droplet":
        b = 0.25 * min(nx, ny, nz) * rng.uniform(0.95, 1.05)
        axes = (b, b, b)
        p.update(fe=CH, sigma=1.0, eta=0.1 * (2.0 * math.sqrt(2.0) / 3.0) / 0.05)
    else:
        b = rng.uniform(0.2, 0.24) * min(ny, nz, nx / 3.0)
        a = b * _axis(case["vr"])
        axes = (a, b, b)
        vol = 4.0 / 3.0 * math.pi * a * b * b
        p.update(fe=HELFRICH, kappa=1.0, k_area=0.05, eta=1.0 / (vol * shear),
                 k_vol=1.0 / (case["dt"] * nx * ny * nz))
    c = np.array([nx / 2.0, H / 2.0, nz / 2.0 if zper else (nz + 1) / 2.0]) + rng.uniform(-1, 1, 3)
    dev = dict(device="cuda", dtype=torch.float64)
    x = (torch.arange(nx, **dev) + 0.5 - c[0])[None, None, :]
    y = (torch.arange(ny, **dev) + 1.0 - c[1])[None, :, None]
    z = (torch.arange(nz, **dev) + (0.5 if zper else 1.0) - c[2])[:, None, None]
    q = [x / axes[0], y / axes[1], z / axes[2]]
    r = torch.sqrt(q[0] ** 2 + q[1] ** 2 + q[2] ** 2).clamp_min(1e-12)
    g = torch.sqrt((q[0] / axes[0]) ** 2 + (q[1] / axes[1]) ** 2 + (q[2] / axes[2]) ** 2) / r
    return torch.tanh((r - 1.0) / g.clamp_min(1e-12) / (math.sqrt(2.0) * eps)), p


def _grid_cases(case):
    """The cases of a batch's grids (one for a batch of one grid)."""
    if "grids" not in case:
        return [case]
    rng = np.random.default_rng(case["sizes"])
    out = []
    for _ in range(case["grids"]):
        n = 8 * rng.integers(case["lo"] // 8, case["hi"] // 8 + 1, 3)
        out.append(_step(None, int(n[0]) * int(rng.integers(1, 3)), int(n[1]), int(n[2]), "mixed",
                         str(rng.choice(["vesicle", "droplet"])), int(rng.choice([DUCT, COUETTE])),
                         case["steps"], cycles=case["cycles"], order=case["order"], dt=case["dt"],
                         vr=float(rng.uniform(0.7, 0.98))))
    return out


def _rhs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen)


def _precision(case):
    return V.VSV_MIXED if case["prec"] == "mixed" else V.VSV_FP64


def _simulation(case, seed, stream=None):
    phi0, p = _scene(case, seed)
    sim = Simulation(case["nx"], case["ny"], case["nz"], 1.0, _precision(case), stream=stream)
    V.vsv_set_flow(sim.g, p["flow"], p["u_max"], p["v_lo"], p["v_hi"], p["eta"], p["rho"])
    V.vsv_set_free_energy(sim.g, p["fe"], p["sigma"], p["kappa"], p["eps"], p["mobility"],
                          p["k_area"], p["k_vol"])
    sp = sim.solver_params()
    sp.tol = case["tol"]
    if case["solver"] == "sor":
        sp.kind, sp.max_cycles, sp.check_every = V.VSV_SOLVER_SOR, 20000, 10
    sp.fixed_cycles, sp.extrapolate = case["cycles"], case["order"]
    V.vsv_set_solver(sim.g, sp)
    return sim, phi0, p


def prepare(case, seed):
    if case["kind"] == "poisson":
        sim = Simulation(case["nx"], case["ny"], case["nz"], 1.0, _precision(case))
        return {"case": case, "sim": sim, "rhs": _rhs(case, seed)}
    if case["kind"] == "batch":
        sims = []
        for i, c in enumerate(_grid_cases(case)):
            stream = torch.cuda.Stream()
            sim, phi0, _ = _simulation(c, seed + 1000 * i, stream)
            stream.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(stream):
                sim.set_phi(phi0)
            stream.synchronize()
            sims.append(sim)
        batch = Batch(sims)
        batch.step(8, case["dt"])   # history and graph, as in a running program
        torch.cuda.synchronize()
        return {"case": case, "sims": sims, "batch": batch}
    sim, phi0, p = _simulation(case, seed)
    if case["kind"] == "adjoint":
        tape = Tape(sim, dict(kind=p["fe"], sigma=p["sigma"], kappa=p["kappa"], eps=p["eps"],
                              mobility=p["mobility"], k_area=p["k_area"], k_vol=p["k_vol"]),
                    every=case["every"])
        tape.set_cycles(case["adj_cycles"])
        target = _scene(case, seed + 1)[0]
        return {"case": case, "tape": tape, "phi0": phi0, "target": target}
    sim.set_phi(phi0)
    return {"case": case, "sim": sim}


# ---------------------------------------------------------------- the calls
def _fields(sim):
    return [sim.field(V.VSV_FIELD_PHI, torch.float64, on_device=True)] + [
        sim.field(V.VSV_FIELD_VEL_X + c, torch.float32, on_device=True) for c in range(3)]


def run(state):
    case = state["case"]
    if case["kind"] == "poisson":
        x = torch.zeros_like(state["rhs"])
        V.vsv_solve_poisson(state["sim"].g, state["rhs"].data_ptr(), x.data_ptr(), V.VSV_DTYPE_F64, 1,
                            (case["per_x"], case["per_y"], case["per_z"]), case["tol"], 200,
                            shift=case["shift"])
        return x
    if case["kind"] == "batch":
        state["batch"].step(case["steps"], case["dt"])
        out = []
        for sim in state["sims"]:
            with torch.cuda.stream(sim.stream):
                out.append(_fields(sim))
        return out
    if case["kind"] == "adjoint":
        tape = state["tape"]
        phi = tape.forward(state["phi0"], case["steps"], case["dt"])
        grad, dkappa, dsigma = tape.backward(phi - state["target"])
        return [phi, grad, dkappa, dsigma]
    sim = state["sim"]
    if case["kind"] == "observe":
        d = sim.diagnostics()
        return {"diag": {k: d[k] for k in ("volume", "area", "reduced_volume", "energy", "com",
                                           "dissipation", "dissipation0", "resistance_rel",
                                           "omega_dev2", "psi_dev2", "max_sigma_t")},
                "profile": sim.stress_profile(),
                "sigma_t": sim.field(V.VSV_FIELD_STRESS_T, torch.float32, on_device=True),
                "fields": _fields(sim)}
    sim.step(case["steps"], case["dt"])
    return _fields(sim)


def work(case):
    if case["kind"] == "batch" and "grids" in case:
        parts = [work(dict(c, kind="batch")) for c in _grid_cases(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n = float(case["nx"] * case["ny"] * case["nz"])
    if case["kind"] == "poisson":
        # rhs and solution; a V(2,2)-cycle contracts by about 30 and does about 90
        # operations per cell
        return {"bytes": 16.0 * n, "flops": 90.0 * n * math.ceil(-math.log(case["tol"]) / math.log(30))}
    if case["kind"] == "observe":
        # phi, omega', psi' (double-word) read; sigma_t, phi and velocity written
        return {"bytes": (7 * 8 + 4 + 8 + 12) * n, "flops": 200.0 * n}
    # a step reads and writes phi, omega' and psi' once (double-word or FP64)
    cycles = case["cycles"] or 3
    step = {"bytes": 2 * 7 * 8 * n, "flops": (6 * 90.0 * cycles + 300.0) * n}
    if case["kind"] == "adjoint":
        # forward, recorded re-run, and a reverse step of the same solves
        k = 2 + 2
        return {"bytes": k * case["steps"] * step["bytes"], "flops": k * case["steps"] * step["flops"]}
    return {"bytes": case["steps"] * step["bytes"] + 20.0 * n, "flops": case["steps"] * step["flops"]}


# ---------------------------------------------------------------- 64-bit values
def _basis(n, per):
    """Orthonormal eigenvectors (columns) and eigenvalues of the 1-D second
    difference: sines (zero ghosts) or the real Fourier basis (periodic)."""
    j = torch.arange(n, dtype=torch.float64, device="cuda")
    if not per:
        k = j + 1.0
        q = math.sqrt(2.0 / (n + 1)) * torch.sin(math.pi / (n + 1) * torch.outer(j + 1.0, k))
        return q, 2.0 * torch.cos(math.pi * k / (n + 1)) - 2.0
    k = torch.div(j + 1.0, 2, rounding_mode="floor")
    ang = 2.0 * math.pi / n * torch.remainder(torch.outer(j, k), n)
    q = torch.where((j % 2 == 1)[None, :], torch.cos(ang), torch.sin(ang))
    q[:, 0] = 1.0
    q = q / torch.linalg.vector_norm(q, dim=0, keepdim=True)
    return q, 2.0 * torch.cos(2.0 * math.pi * k / n) - 2.0


class _Poisson:
    """x with (L - shift) x = b for zero ghosts / periodic axes (h = 1)."""

    def __init__(self, nx, ny, nz, per):
        (self.qx, lx), (self.qy, ly), (self.qz, lz) = (_basis(n, p) for n, p in zip((nx, ny, nz), per))
        self.lam = lz[:, None, None] + ly[None, :, None] + lx[None, None, :]

    def __call__(self, b, shift=0.0):
        t = torch.einsum("zyx,xa->zya", b, self.qx)
        t = torch.einsum("zya,yb->zba", t, self.qy)
        t = torch.einsum("zba,zc->cba", t, self.qz) / (self.lam - shift)
        t = torch.einsum("cba,zc->zba", t, self.qz)
        t = torch.einsum("zba,yb->zya", t, self.qy)
        return torch.einsum("zya,xa->zyx", t, self.qx)


def _sh(u, axis, d, ghost):
    """u at the neighbour d along axis; ghost: "per", "mirror" or "zero"."""
    if ghost == "per":
        return torch.roll(u, -d, axis)
    n = u.shape[axis]
    edge = u.narrow(axis, n - 1 if d > 0 else 0, 1)
    edge = edge if ghost == "mirror" else torch.zeros_like(edge)
    return (torch.cat([u.narrow(axis, 1, n - 1), edge], axis) if d > 0
            else torch.cat([edge, u.narrow(axis, 0, n - 1)], axis))


def _d(u, axis, ghost):
    return 0.5 * (_sh(u, axis, 1, ghost) - _sh(u, axis, -1, ghost))


class _Reference:
    """The discrete step in 64 bits (h = 1): forward Euler for phi, then the
    vorticity and the stream-vector problems solved exactly."""

    def __init__(self, p):
        self.p = p
        self.gm = ("per", "mirror", "per" if p["zper"] else "mirror")   # scalars: x, y, z
        self.g0 = ("per", "zero", "per" if p["zper"] else "zero")       # flow perturbation
        self.poisson = _Poisson(p["nx"], p["ny"], p["nz"], (1, 0, int(p["zper"])))
        self.base()

    def lap(self, u):
        s = sum(_sh(u, 2 - a, d, self.gm[a]) for a in range(3) for d in (1, -1))
        return s - 6.0 * u

    def grad(self, u):
        return [_d(u, 2 - a, self.gm[a]) for a in range(3)]

    def base(self):
        """Body-free omega, psi on the (z, y) nodes -1 .. n (wall data on the
        ring) and the velocity of the cells."""
        p = self.p
        ny, nz, H = p["ny"], p["nz"], p["ny"] + 1.0
        y = torch.arange(ny + 2, dtype=torch.float64, device="cuda")[None, :].expand(nz + 2, -1)
        zero = torch.zeros(nz + 2, ny + 2, dtype=torch.float64, device="cuda")
        self.om0, self.ps0 = [zero.clone() for _ in range(3)], [zero.clone() for _ in range(3)]
        if p["flow"] == COUETTE:
            dv = p["v_hi"] - p["v_lo"]
            self.ps0[2] = p["v_lo"] * y + dv * y * y / (2.0 * H)
            self.om0[2] = zero - dv / H
        elif p["flow"] == PLANAR:
            u = 4.0 * p["u_max"] / (H * H)
            self.ps0[2] = u * (H * y * y / 2.0 - y ** 3 / 3.0)
            self.om0[2] = -u * (H - 2.0 * y)
        else:
            s = _Poisson(1, ny, nz, (1, 0, 0))
            u0 = s(-torch.ones(nz, ny, 1, dtype=torch.float64, device="cuda"))[:, :, 0]
            u0 = u0 * (p["u_max"] / u0.max())
            chi = s(u0[:, :, None])[:, :, 0]

            def one(a, b):
                return (4.0 * a - b) / 2.0
            for f, omega in ((u0, True), (chi, False)):
                sg = 1.0 if omega else -1.0
                ry, rz = (self.om0[1], self.om0[2]) if omega else (self.ps0[1], self.ps0[2])
                rz[1:-1, 0], rz[1:-1, -1] = -sg * one(f[:, 0], f[:, 1]), sg * one(f[:, -1], f[:, -2])
                ry[0, 1:-1], ry[-1, 1:-1] = sg * one(f[0], f[1]), -sg * one(f[-1], f[-2])

            def fill(ring, rhs):
                b = rhs.clone()
                b[:, 0] -= ring[1:-1, 0]
                b[:, -1] -= ring[1:-1, -1]
                b[0] -= ring[0, 1:-1]
                b[-1] -= ring[-1, 1:-1]
                ring[1:-1, 1:-1] = s(b[:, :, None])[:, :, 0]
            for c in (1, 2):
                fill(self.om0[c], torch.zeros(nz, ny, dtype=torch.float64, device="cuda"))
                fill(self.ps0[c], -self.om0[c][1:-1, 1:-1])
        dy = 0.5 * (self.ps0[2][1:-1, 2:] - self.ps0[2][1:-1, :-2])
        dz = 0.5 * (self.ps0[1][2:, 1:-1] - self.ps0[1][:-2, 1:-1])
        self.v0 = (dy - dz)[:, :, None]   # x component; the others vanish

    def velocity(self, ps):
        d = [[_d(ps[c], 2 - a, self.g0[a]) for a in range(3)] for c in range(3)]
        return [d[2][1] - d[1][2] + self.v0, d[0][2] - d[2][0], d[1][0] - d[0][1]]

    def volume_area(self, phi):
        eps = self.p["eps"]
        g = self.grad(phi)
        dens = 0.5 * eps * (g[0] ** 2 + g[1] ** 2 + g[2] ** 2) + (phi * phi - 1.0) ** 2 / (4.0 * eps)
        return 0.5 * (1.0 - phi).sum(), 3.0 / (2.0 * math.sqrt(2.0)) * dens.sum()

    def g(self, phi):
        return phi ** 3 - phi - self.p["eps"] ** 2 * self.lap(phi)

    def mu(self, phi, gamma, kappa, sigma):
        p = self.p
        if p["fe"] == CH:
            return phi ** 3 - phi - sigma * self.lap(phi)
        g = self.g(phi)
        cf2 = 3.0 * math.sqrt(2.0) * kappa / (4.0 * p["eps"] ** 3)
        return (cf2 * ((3.0 * phi * phi - 1.0) * g - p["eps"] ** 2 * self.lap(g)) - gamma * self.lap(phi)
                + sigma * (3.0 / (2.0 * math.sqrt(2.0) * p["eps"])) * g)

    def solve(self, phi, mu, om=None):
        p = self.p
        a, b = self.grad(phi), self.grad(mu)
        f = [(a[1] * b[2] - a[2] * b[1]) / p["eta"], (a[2] * b[0] - a[0] * b[2]) / p["eta"],
             (a[0] * b[1] - a[1] * b[0]) / p["eta"]]
        s = p["rho"] / (p["eta"] * p["dt"]) if om is not None else 0.0
        om = [self.poisson(f[c] - s * om[c], s) if s else self.poisson(f[c]) for c in range(3)]
        return om, [self.poisson(-om[c]) for c in range(3)]

    def run(self, phi, steps, kappa=None, sigma=None):
        """(phi, omega', psi') after `steps` steps from phi."""
        p = self.p
        kappa = p["kappa"] if kappa is None else kappa
        sigma = p["sigma"] if sigma is None else sigma
        v_ref, a_ref = self.volume_area(phi)
        vol = v_ref
        mu = self.mu(phi, 0.0, kappa, sigma)
        om, ps = self.solve(phi, mu)
        for _ in range(steps):
            v, g = self.velocity(ps), self.grad(phi)
            lam = p["k_vol"] * (vol - v_ref)
            phi = phi + p["dt"] * (p["mobility"] * (self.lap(mu) + lam)
                                   - (v[0] * g[0] + v[1] * g[1] + v[2] * g[2]))
            vol, area = self.volume_area(phi)
            gamma = p["k_area"] * (area - a_ref) * 3.0 * p["eps"] / (2.0 * math.sqrt(2.0))
            mu = self.mu(phi, gamma, kappa, sigma)
            om, ps = self.solve(phi, mu, om)
        return phi, om, ps


def _exact_observe(ref, phi):
    p = ref.p
    _, om, ps = ref.run(phi, 0)
    v = ref.velocity(ps)
    vol, area = ref.volume_area(phi)

    def strain(v):
        """2 e_ij of a velocity with the walls' speeds on the wall nodes"""
        def d(u, c, a):
            t = _d(u, 2 - a, ref.g0[a])
            if a == 1 and c == 0:
                t[:, 0, :] -= 0.5 * p["v_lo"]
                t[:, -1, :] += 0.5 * p["v_hi"]
            return t
        g = [[d(v[i], i, a) for a in range(3)] for i in range(3)]
        return [[g[i][j] + g[j][i] for j in range(3)] for i in range(3)]
    e = strain(v)
    zero = torch.zeros_like(phi)
    e0 = strain([ref.v0 + zero, zero, zero])
    diss = [0.5 * p["eta"] * sum(x.square().sum() for r in t for x in r) for t in (e, e0)]
    sig = p["eta"] * torch.sqrt(e[0][1] ** 2 + e[1][2] ** 2 + e[0][2] ** 2)
    if p["fe"] == HELFRICH:
        energy = 3.0 * math.sqrt(2.0) * p["kappa"] / (8.0 * p["eps"] ** 3) * ref.g(phi).square().sum()
    else:
        grad2 = sum((_sh(phi, 2 - a, 1, ref.gm[a]) - phi).square().sum() for a in range(3))
        energy = 0.25 * (phi * phi - 1.0).square().sum() + 0.5 * p["sigma"] * grad2
    w = 0.5 * (1.0 - phi)
    off = (0.5, 1.0, 0.5 if p["zper"] else 1.0)
    com = []
    for a in range(3):
        x = torch.arange(phi.shape[2 - a], dtype=torch.float64, device="cuda") + off[a]
        com.append(float((w.sum([b for b in range(3) if b != 2 - a]) * x).sum() / w.sum()))
    diag = {"volume": float(vol), "area": float(area),
            "reduced_volume": float(vol / (4.0 / 3.0 * math.pi * (area / (4.0 * math.pi)) ** 1.5)),
            "energy": float(energy), "com": com, "dissipation": float(diss[0]),
            "dissipation0": float(diss[1]), "resistance_rel": float((diss[0] - diss[1]) / diss[1]),
            "omega_dev2": float(sum(o.square().sum() for o in om)),
            "psi_dev2": float(sum(s.square().sum() for s in ps)), "max_sigma_t": float(sig.max())}
    return {"diag": diag, "profile": (p["eta"] * e[0][1]).mean(dim=(0, 2)).cpu().numpy(),
            "sigma_t": sig, "fields": [phi] + v}


def exact(case, seed):
    if case["kind"] == "poisson":
        per = (case["per_x"], case["per_y"], case["per_z"])
        return _Poisson(case["nx"], case["ny"], case["nz"], per)(_rhs(case, seed), case["shift"])
    if case["kind"] == "batch":
        out = []
        for i, c in enumerate(_grid_cases(case)):
            phi0, p = _scene(c, seed + 1000 * i)
            ref = _Reference(p)
            phi, _, ps = ref.run(phi0, 8 + case["steps"])
            out.append([phi] + ref.velocity(ps))
        return out
    phi0, p = _scene(case, seed)
    ref = _Reference(p)
    if case["kind"] == "observe":
        return _exact_observe(ref, phi0)
    if case["kind"] == "step":
        phi, _, ps = ref.run(phi0, case["steps"])
        return [phi] + ref.velocity(ps)
    phi0.requires_grad_(True)
    one = dict(dtype=torch.float64, device="cuda", requires_grad=True)
    kappa, sigma = torch.tensor(p["kappa"], **one), torch.tensor(p["sigma"], **one)
    phi, _, _ = ref.run(phi0, case["steps"], kappa, sigma)
    target = _scene(case, seed + 1)[0]
    g = torch.autograd.grad(phi, (phi0, kappa, sigma), grad_outputs=(phi - target).detach(),
                            allow_unused=True)
    g = [torch.zeros((), dtype=torch.float64) if t is None else t.detach() for t in g]
    return [phi.detach(), g[0], float(g[1]), float(g[2])]
