"""Performance cases of the particle-in-cell step: what a user of this package
has it do, through its public entry points, over the sizes it is used at.

A case's `kind` names the call:
  run          whole steps of one instance (Sim.step), then the tallies and the
               grid fields that a run writes out
  batch        the same for uneven instances that advance together
  restart      a checkpoint taken up again for one step, particles read back
  poisson      one field solve of a given charge density (Sim.solve_poisson)
  adjoint      the gradient of window means by the reverse sweep (Sim.adjoint)
  sensitivity  the same window's Jacobian in forward mode (Sim.sensitivity)
  deposit      charge weighing of caller-owned particles (apic_deposit_static)

Grids are counted in cells, units are those of include/apic.h.  Quantities of
the FP32 form come back as FP32, the precision of its particles; those of the
FP64 form, and the field solve that is refined in FP64, as FP64.
"""
import ctypes as C
import math

import numpy as np
import torch

import paper_2307_11107_gb300 as apic
from paper_2307_11107_gb300 import _abi
from paper_2307_11107_gb300.workloads import batched_48

ELECTRON = dict(q=-1.0, m=1.0, T=1.0)


def _run(name, n1, n2, electrons, ions, steps, **kw):
    c = dict(name=name, kind="run", precision="fp32", n1=n1, n2=n2, electrons=electrons, ions=ions, steps=steps,
             alpha=0.15, x1_out=-0.05, phi_g=-2.5, B=1.0, dt=0.1, Ti=0.5, sort_interval=8, poisson_tol=1e-10,
             poisson_max_iter=20, poisson_guess=0)
    c.update(kw)
    return c


def listed():
    return [
        # a program that follows the grain step by step (charge, force, bins
        # after every step) on the smallest grid the tests use: launch latency
        _run("follow_32x16", 32, 16, 4000, 4000, 1, B=0.5, x1_out=-0.1, sort_interval=0),
        # the spherical grain in FP64, as the tests and the parity runs have it
        _run("sphere_fp64_64x32", 64, 32, 100000, 100000, 20, precision="fp64", alpha=0.0, x1_out=-0.1, B=0.0,
             Ti=1.0, sort_interval=0, poisson_tol=1e-13, poisson_max_iter=40),
        # an isolated, strongly shaped grain on a grid that is no power of two,
        # with unequal odd particle counts
        _run("floating_264x92", 264, 92, 345679, 123457, 10, alpha=-0.2, x1_out=-0.08, B=0.5, sort_interval=5,
             floating=True),
        # the dipole-shaped grain, a production run's steps
        _run("dipole_256x128_2e7", 256, 128, 10_000_000, 10_000_000, 16, poisson_guess=1),
        # the same form at scale: the benchmark's workload
        _run("dipole_1024x512_1e8", 1024, 512, 50_000_000, 50_000_000, 16, alpha=0.225, poisson_max_iter=30),
        # a reference run in FP64 beside the production one
        _run("dipole_fp64_256x128", 256, 128, 1_000_000, 1_000_000, 8, precision="fp64", poisson_tol=1e-12,
             poisson_max_iter=60),
        # ions alone in Boltzmann electrons, the long time step of ion dynamics
        _run("boltzmann_256x128", 256, 128, 0, 10_000_000, 4, dt=1.0, boltzmann=True, poisson_max_iter=30,
             poisson_guess=1),
        # a parameter scan: 48 uneven instances in one launch per phase
        dict(name="scan_48", kind="batch", instances=48, scale=1.0, scan_seed=2, steps=16),
        # a checkpoint taken up again for one step, particles read back
        dict(name="restart_fp32_64x32", kind="restart", precision="fp32", n1=64, n2=32, n=20000, alpha=0.15,
             x1_out=-0.1, phi_g=-2.5, B=1.0, dt=0.1),
        # the field of a given density
        dict(name="poisson_512x256", kind="poisson", precision="fp32", n1=512, n2=256, alpha=0.225, x1_out=-0.05,
             phi_g=-2.5, tol=1e-10),
        # shape, potential and magnetic-field gradients of a 10-step window
        dict(name="adjoint_256x128", kind="adjoint", precision="fp32", n1=256, n2=128, n=1_000_000, steps=10,
             alpha=0.15, x1_out=-0.05, phi_g=-2.5, B=1.0, dt=0.1),
        # density of particles that another program holds
        dict(name="deposit_512x256_1e7", kind="deposit", n1=512, n2=256, n=10_000_000, alpha=0.15, x1_out=-0.05),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, n1_lo, n1_hi):
    """A grid that multigrid coarsening takes (down to a level of at most 2200
    unknowns): 64 x 24, 264 x 92, 768 x 400 and the like."""
    while True:
        n1, n2 = _log_int(rng, n1_lo, n1_hi), _log_int(rng, 16, 512)
        if not 1.0 <= n1 / n2 <= 4.0:
            continue
        k = 0  # halvings until the level is small
        while (n1 / 2 ** k - 1) * (n2 / 2 ** k + 1) > 2000:
            k += 1
        n1, n2 = max(1, n1 >> k) << k, max(1, n2 >> k) << k
        if n1 >= n1_lo and n2 >= 16:
            return n1, n2


def draw(rng):
    kind = rng.choice(["run"] * 8 + ["run64", "batch", "restart", "poisson", "poisson", "adjoint", "sensitivity",
                                     "deposit"])
    phys = dict(alpha=round(rng.uniform(-0.24, 0.24), 4), x1_out=rng.choice([-0.05, -0.08, -0.1]),
                phi_g=round(rng.uniform(-4.0, -1.0), 3), B=rng.choice([0.0, 0.5, 1.0]))
    if kind == "run":
        n1, n2 = _grid(rng, 32, 1024)
        ne = _log_int(rng, 4000, 30_000_000)
        c = _run("", n1, n2, ne, max(1000, int(ne * rng.choice([1.0, 1.0, 0.37]))), rng.choice([1, 5, 8, 13, 16]),
                 sort_interval=rng.choice([0, 4, 8, 12]) if ne < 200_000 else rng.choice([4, 8, 12]),
                 Ti=rng.choice([0.1, 0.5, 1.0]), poisson_max_iter=30, poisson_guess=rng.choice([0, 1]), **phys)
        if rng.random() < 0.2:
            c["floating"] = True
    elif kind == "run64":
        n1, n2 = _grid(rng, 32, 256)
        ne = _log_int(rng, 4000, 1_000_000)
        c = _run("", n1, n2, ne, ne, rng.choice([1, 5, 8, 20]), precision="fp64",
                 sort_interval=rng.choice([0, 8]), poisson_tol=1e-12, poisson_max_iter=60, **phys)
    elif kind == "batch":
        c = dict(kind="batch", instances=rng.randint(2, 24), scale=round(math.exp(rng.uniform(math.log(0.02), 0.0)), 3),
                 scan_seed=rng.randint(3, 999), steps=rng.choice([4, 8, 16]))
    elif kind == "restart":
        n1, n2 = _grid(rng, 32, 128)
        c = dict(kind="restart", precision=rng.choice(["fp32", "fp64"]), n1=n1, n2=n2, n=_log_int(rng, 2000, 60000),
                 dt=0.1, **phys)
    elif kind == "poisson":
        n1, n2 = _grid(rng, 32, 1024)
        c = dict(kind="poisson", precision="fp32" if n1 > 256 else rng.choice(["fp32", "fp32", "fp64"]), n1=n1, n2=n2,
                 tol=1e-10, **phys)
        del c["B"]
    elif kind in ("adjoint", "sensitivity"):
        n1, n2 = _grid(rng, 32, 256)
        c = dict(kind=kind, precision=rng.choice(["fp32", "fp64"]), n1=n1, n2=n2, n=_log_int(rng, 10_000, 1_000_000),
                 steps=rng.choice([3, 5, 10]), dt=0.1, **phys)
    else:
        n1, n2 = _grid(rng, 32, 1024)
        c = dict(kind="deposit", n1=n1, n2=n2, n=_log_int(rng, 10_000, 20_000_000), alpha=phys["alpha"],
                 x1_out=phys["x1_out"])
    c.pop("name", None)
    return c


# ---- preparation: the simulation object with its plasma loaded ----
def _instance(c, species, seed, **kw):
    return dict(alpha=c["alpha"], x1_out=c["x1_out"], phi_g=c["phi_g"], phi_out=0.0, B=c.get("B", 0.0),
                dt=c.get("dt", 0.1), n1=c["n1"], n2=c["n2"], species=species, seed=seed, precision=c["precision"], **kw)


def _ion(T):
    return dict(q=1.0, m=1836.0, T=T)


def _states(c, seed):
    """Explicit states, n rows (x1, x2, vR, vZ, vTheta) per species: uniform in
    physical volume, Maxwellian, as FP32 values (both forms take them exactly)."""
    rng = np.random.default_rng(seed)
    out = []
    for vth in (1.0, math.sqrt(0.5 / 1836.0)):
        x2 = rng.uniform(-0.999, 0.999, c["n"])
        rg = (1 + np.sqrt(1 + 4 * c["alpha"] * x2)) / 2
        ro = -(1 + np.sqrt(1 - 4 * c["alpha"] * c["x1_out"] * x2)) / (2 * c["x1_out"])
        r = np.cbrt(rg ** 3 + rng.uniform(0.001, 0.999, c["n"]) * (ro ** 3 - rg ** 3))
        x1 = -(1 + c["alpha"] * x2 / r) / r
        v = rng.standard_normal((c["n"], 3)) * vth
        out.append(np.column_stack([x1, x2, v]).astype(np.float32).astype(np.float64))
    return out


def _density(c, seed):
    """A charge density as particles give it: smooth, with shot noise."""
    rng = np.random.default_rng(seed)
    x1 = np.linspace(-1.0, c["x1_out"], c["n1"] + 1)[:, None]
    x2 = np.linspace(-1.0, 1.0, c["n2"] + 1)[None, :]
    a, b = rng.uniform(0.2, 0.5), rng.uniform(-0.3, 0.3)
    return a * np.exp(-6.0 * (x1 + 1.0)) * (1.0 + b * x2) + 0.03 * rng.standard_normal((c["n1"] + 1, c["n2"] + 1))


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "run":
        species, counts = [], []
        if c["electrons"]:
            species.append(dict(ELECTRON, n_init=c["electrons"]))
            counts.append(c["electrons"])
        species.append(dict(_ion(c["Ti"]), n_init=c["ions"]))
        counts.append(c["ions"])
        opt = {k: c[k] for k in ("sort_interval", "poisson_tol", "poisson_max_iter", "poisson_guess", "floating",
                                 "boltzmann") if k in c}
        if c.get("boltzmann"):
            opt["newton_iters"] = 8
        sim = apic.Sim(_instance(c, species, seed, history_cap=64, **opt))
        for s, n in enumerate(counts):
            sim.load_volume(s, n)
        return dict(case=c, sim=sim)
    if kind == "batch":
        cfgs = [dict(w, seed=seed, history_cap=64) for w in batched_48(c["scan_seed"], c["scale"])[:c["instances"]]]
        sim = apic.Sim(cfgs)
        for k, w in enumerate(cfgs):
            for s, sp in enumerate(w["species"]):
                sim.load_volume(s, sp["n_init"], instance=k)
        return dict(case=c, sim=sim)
    if kind == "restart":
        species = [dict(ELECTRON, n_init=c["n"]), dict(_ion(0.5), n_init=c["n"])]
        sim = apic.Sim(_instance(c, species, 1, no_inject=True, history_cap=64, poisson_tol=1e-12, poisson_max_iter=60))
        for s, st in enumerate(_states(c, seed)):
            sim.add_particles(s, st)
        return dict(case=c, sim=sim, saved=sim.checkpoint())
    if kind == "poisson":
        species = [dict(ELECTRON, n_init=1000), dict(_ion(0.5), n_init=1000)]
        sim = apic.Sim(_instance(c, species, 1, poisson_tol=c["tol"], poisson_max_iter=60))
        return dict(case=c, sim=sim, rho=_density(c, seed))
    if kind in ("adjoint", "sensitivity"):
        species = [dict(ELECTRON, n_init=c["n"]), dict(_ion(0.5), n_init=c["n"])]
        tol = 1e-10 if c["precision"] == "fp32" else 1e-12
        sim = apic.Sim(_instance(c, species, seed, history_cap=64, poisson_tol=tol, poisson_max_iter=60))
        for s in (0, 1):
            sim.load_volume(s, c["n"])
        return dict(case=c, sim=sim, w=np.array([1.0, 1.0, 0.5, 2.0, 0.1]))
    x1, x2 = _positions(c, seed)
    V = _volumes(c)
    return dict(case=c, lib=apic.load(), x1=x1, x2=x2, V=V, rho=torch.empty_like(V))


# ---- one pass ----
def _real(c, a):
    return a.astype(np.float32) if c.get("precision", "fp32") == "fp32" else a


def _rows(c, st):
    """The particles still there, in the fixed table of n rows a program keeps (the rest zero)."""
    out = np.zeros((c["n"], 5))
    out[:len(st)] = st
    return out


def _written(c, sim, k=0):
    """What a run writes out after its steps."""
    t = sim.tallies(k)
    counts = np.array([list(s.values()) for s in t["counts"]], dtype=np.int64)
    return dict(bins=_real(c, t["bins"]), counts=counts, history=_real(c, t["history"][-c["steps"]:]),
                grain=_real(c, np.array([t["Q"], t["FZ"]])), phi=_real(c, sim.field("phi", k)),
                rho=_real(c, sim.field("rho", k)))


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "deposit":
        grid = _abi.Grid(c["n1"], c["n2"], c["x1_out"])
        s = torch.cuda.current_stream()
        rc = state["lib"].apic_deposit_static(C.byref(grid), state["x1"].data_ptr(), state["x2"].data_ptr(), c["n"],
                                              -1.0 / c["n"], state["V"].data_ptr(), state["rho"].data_ptr(),
                                              C.c_void_p(s.cuda_stream))
        if rc != 0:
            raise RuntimeError("apic_deposit_static: %d" % rc)
        return state["rho"]
    sim = state["sim"]
    if kind == "run":
        sim.step(c["steps"])
        return _written(c, sim)
    if kind == "batch":
        sim.step(c["steps"])
        out = [_written(c, sim, k) for k in range(sim.n_inst)]
        return {key: np.concatenate([o[key].reshape(-1) for o in out]) for key in out[0]}
    if kind == "restart":
        sim.restore(state["saved"])
        sim.step(1)
        return dict(phi=_real(c, sim.field("phi")), rho=_real(c, sim.field("rho")),
                    electrons=_real(c, _rows(c, sim.particles(0))), ions=_real(c, _rows(c, sim.particles(1))))
    if kind == "poisson":
        return sim.solve_poisson(state["rho"])
    if kind == "adjoint":
        grad, values = sim.adjoint(c["steps"], state["w"], values=True)
        return dict(grad=_real(c, grad), values=_real(c, values), phi=_real(c, sim.field("phi")),
                    rho=_real(c, sim.field("rho")))
    r = sim.sensitivity(c["steps"])
    return dict(jacobian=_real(c, r["jacobian"]), values=_real(c, r["values"]), phi=_real(c, sim.field("phi")),
                rho=_real(c, sim.field("rho")))


# ---- what a pass cannot do without ----
def _push_work(c, particles, steps):
    """Per step: the particles' five components read and written, 127 operations
    for each (FP32 count of the equations of motion, gather and weighing); the
    density written and the potential written and read on the nodes."""
    b = 40.0 if c.get("precision", "fp32") == "fp32" else 80.0
    nodes = (c["n1"] + 1.0) * (c["n2"] + 1.0)
    return steps * (b * particles + 24.0 * nodes), steps * (127.0 * particles + 22.0 * nodes)


def work(case):
    c, kind = case, case["kind"]
    if kind == "deposit":
        nodes = (c["n1"] + 1.0) * (c["n2"] + 1.0)
        return {"bytes": 16.0 * c["n"] + 16.0 * nodes, "flops": 16.0 * c["n"] + 2.0 * nodes}
    if kind == "poisson":
        nodes = (c["n1"] + 1.0) * (c["n2"] + 1.0)
        return {"bytes": 16.0 * nodes, "flops": 22.0 * nodes}
    if kind == "batch":
        b = f = 0.0
        for w in batched_48(c["scan_seed"], c["scale"])[:c["instances"]]:
            x, y = _push_work(w, 2.0 * w["species"][0]["n_init"], c["steps"])
            b, f = b + x, f + y
        return {"bytes": b, "flops": f}
    if kind == "run":
        b, f = _push_work(c, float(c["electrons"] + c["ions"]), c["steps"])
    elif kind == "restart":
        b, f = _push_work(c, 2.0 * c["n"], 1)
    elif kind == "adjoint":  # forward, then backward: each state read again, its adjoint read and written
        b, f = _push_work(c, 2.0 * c["n"], c["steps"])
        b, f = 2.5 * b, 4.0 * f
    else:  # the state and three directions of it
        b, f = _push_work(c, 2.0 * c["n"], c["steps"])
        b, f = 4.0 * b, 4.0 * f
    return {"bytes": b, "flops": f}


# ---- plain FP64 values, from the equations ----
def _radius(al, x1, x2):
    """Eq. 3."""
    return -(1.0 + torch.sqrt(1.0 - 4.0 * al * x1 * x2)) / (2.0 * x1)


def _positions(c, seed):
    """Positions uniform in physical volume, in no order."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    u = torch.rand((2, c["n"]), dtype=torch.float64, device="cuda", generator=g)
    x2 = 2.0 * u[0] - 1.0
    one = torch.ones((), dtype=torch.float64, device="cuda")
    rg, ro = _radius(c["alpha"], -one, x2), _radius(c["alpha"], c["x1_out"] * one, x2)
    r = (rg ** 3 + u[1] * (ro ** 3 - rg ** 3)) ** (1.0 / 3.0)
    return (-(1.0 + c["alpha"] * x2 / r) / r).clamp_(-1.0, c["x1_out"]).contiguous(), x2.contiguous()


def _nodes(c, dev):
    x1 = torch.linspace(-1.0, c["x1_out"], c["n1"] + 1, dtype=torch.float64, device=dev)
    x2 = torch.linspace(-1.0, 1.0, c["n2"] + 1, dtype=torch.float64, device=dev)
    return x1[:, None], x2[None, :], (c["x1_out"] + 1.0) / c["n1"], 2.0 / c["n2"]


def _volumes(c):
    """Node volumes by the trapezoid rule on Eq. 5."""
    x1, x2, h1, h2 = _nodes(c, "cuda")
    r = _radius(c["alpha"], x1, x2)
    V = 2.0 * math.pi * r ** 4 / (1.0 + 2.0 * c["alpha"] * x2 / r) * (h1 * h2)
    V[[0, -1], :] *= 0.5
    V[:, [0, -1]] *= 0.5
    return V.contiguous()


def _cells(c, x1, x2):
    h1, h2 = (c["x1_out"] + 1.0) / c["n1"], 2.0 / c["n2"]
    u1, u2 = (x1 + 1.0) / h1, (x2 + 1.0) / h2
    i, j = u1.floor().clamp(0, c["n1"] - 1), u2.floor().clamp(0, c["n2"] - 1)
    f1, f2 = (u1 - i).clamp(0, 1), (u2 - j).clamp(0, 1)
    k = (i * (c["n2"] + 1) + j).long()
    return [(k, (1 - f1) * (1 - f2)), (k + c["n2"] + 1, f1 * (1 - f2)), (k + 1, (1 - f1) * f2),
            (k + c["n2"] + 2, f1 * f2)]


def _weigh(c, x1, x2):
    out = torch.zeros((c["n1"] + 1) * (c["n2"] + 1), dtype=torch.float64, device=x1.device)
    for k, w in _cells(c, x1, x2):
        out += torch.bincount(k, weights=w, minlength=out.numel())
    return out.view(c["n1"] + 1, c["n2"] + 1)


def _hat_volumes(c, dev):
    """Integrals of each node's bilinear weight over Eq. 5's volume element
    (eight Gauss points a cell and direction)."""
    gx, gw = np.polynomial.legendre.leggauss(8)
    x1, x2, h1, h2 = _nodes(c, dev)
    V = torch.zeros((c["n1"] + 1, c["n2"] + 1), dtype=torch.float64, device=dev)
    for a, wa in zip(0.5 * (gx + 1), 0.5 * gw):
        for b, wb in zip(0.5 * (gx + 1), 0.5 * gw):
            p, q = x1[:-1] + a * h1, x2[:, :-1] + b * h2
            r = _radius(c["alpha"], p, q)
            m = 2.0 * math.pi * r ** 4 / (1.0 + 2.0 * c["alpha"] * q / r) * (wa * wb * h1 * h2)
            V[:-1, :-1] += m * ((1 - a) * (1 - b))
            V[1:, :-1] += m * (a * (1 - b))
            V[:-1, 1:] += m * ((1 - a) * b)
            V[1:, 1:] += m * (a * b)
    return V


def _field(c, rho):
    """Eqs. 6-7 by second-order differences (one-sided at the poles), by block
    elimination over the rows of x1."""
    dev, al, n1, n2 = rho.device, c["alpha"], c["n1"], c["n2"]
    x1, x2, h1, h2 = _nodes(c, dev)
    N = n2 + 1
    j = torch.arange(1, n2, device=dev)
    s2 = ((1 - x2) * (1 + x2))[0]

    def row(i):
        """Blocks of row i on rows i - 1, i, i + 1, divided by the x1 coefficient."""
        r = _radius(al, x1[i], x2[0])
        a1 = ((r + 2 * al * x2[0]) ** 2 + al * al * s2) / r ** 6 / h1 ** 2
        a2, d = s2 / r ** 2 / h2 ** 2, -2 * al * s2 / r ** 4 / (4 * h1 * h2)
        e = -2 * x2[0] / r ** 2 / (2 * h2)
        lo, mid, hi = (torch.zeros((N, N), dtype=torch.float64, device=dev) for _ in range(3))
        lo.diagonal().add_(a1)
        hi.diagonal().add_(a1)
        mid.diagonal().sub_(2 * a1)
        mid[j, j] -= 2 * a2[j]
        mid[j, j - 1] += (a2 - e)[j]
        mid[j, j + 1] += (a2 + e)[j]
        hi[j, j + 1] += d[j]
        hi[j, j - 1] -= d[j]
        lo[j, j - 1] += d[j]
        lo[j, j + 1] -= d[j]
        mid[0, :3] += e[0] * torch.tensor([-3.0, 4.0, -1.0], dtype=torch.float64, device=dev)
        mid[n2, n2 - 2:] += e[n2] * torch.tensor([1.0, -4.0, 3.0], dtype=torch.float64, device=dev)
        return lo / a1[:, None], mid / a1[:, None], hi / a1[:, None], -rho[i] / a1

    phi = torch.zeros((n1 + 1, N), dtype=torch.float64, device=dev)
    phi[0] = c["phi_g"]
    up, f = [], []
    for i in range(1, n1):
        lo, mid, hi, b = row(i)
        if i == 1:
            b = b - lo @ phi[0]
        else:
            mid, b = mid - lo @ up[-1], b - lo @ f[-1]
        x = torch.linalg.solve(mid, torch.cat([hi, b[:, None]], 1))
        up.append(x[:, :N].contiguous())
        f.append(x[:, N].contiguous())
    for i in range(n1 - 1, 0, -1):
        phi[i] = f[i - 1] - up[i - 1] @ phi[i + 1]
    return phi


def _slope(p, h, dim):
    """Central differences, one-sided of second order at the two ends."""
    p = p.movedim(dim, 0)
    g = torch.empty_like(p)
    g[1:-1] = (p[2:] - p[:-2]) / (2 * h)
    g[0] = (-3 * p[0] + 4 * p[1] - p[2]) / (2 * h)
    g[-1] = (3 * p[-1] - 4 * p[-2] + p[-3]) / (2 * h)
    return g.movedim(0, dim)


def _moved(c, G1, G2, q, m, st):
    """One step of each particle (Eqs. 3, 8, 9, 10 and 2); the rows that stay
    between the grain and the outer surface."""
    al, dt = c["alpha"], c["dt"]
    x1, x2, vR, vZ, vT = st.T
    r = _radius(al, x1, x2)
    s = torch.sqrt((1 - x2) * (1 + x2))
    g1 = sum(w * G1.reshape(-1)[k] for k, w in _cells(c, x1, x2))
    g2 = sum(w * G2.reshape(-1)[k] for k, w in _cells(c, x1, x2))
    ER = -(s * (r + 3 * al * x2) / r ** 3 * g1 - x2 * s / r * g2)
    EZ = -((r * x2 + al * (3 * x2 ** 2 - 1)) / r ** 3 * g1 + s * s / r * g2)
    h = 0.5 * q / m * dt
    a, b, z = vR + h * ER, vT, vZ + h * EZ
    t = -h * c["B"]
    a2, b2 = a + b * t, b - a * t
    a, b = a + b2 * (2 * t / (1 + t * t)) + h * ER, b - a2 * (2 * t / (1 + t * t))
    z = z + h * EZ
    X, Y, Z = r * s + a * dt, b * dt, r * x2 + z * dt
    Rn = torch.sqrt(X * X + Y * Y)
    rn = torch.sqrt(Rn * Rn + Z * Z)
    y2 = Z / rn
    y1 = -(1 + al * y2 / rn) / rn
    live = (rn >= (1 + torch.sqrt(1 + 4 * al * y2)) / 2) & (y1 <= c["x1_out"])
    return torch.stack([y1, y2, (X * a + Y * b) / Rn, z, (X * b - Y * a) / Rn], 1)[live]


def exact(case, seed):
    """Plain FP64 values of the calls that are one evaluation: a weighing, a
    field, one step of given particles.  A run of many steps draws its plasma
    and its injection from the library's generator and amplifies rounding: it
    has no such value here."""
    c, kind = case, case["kind"]
    if kind == "deposit":
        x1, x2 = _positions(c, seed)
        return -1.0 / c["n"] * _weigh(c, x1, x2) / _volumes(c)
    if kind == "poisson":
        return _field(c, torch.tensor(_density(c, seed), device="cuda"))
    if kind == "restart":
        st = [torch.tensor(s, device="cuda") for s in _states(c, seed)]
        x2 = torch.linspace(-1.0, 1.0, 4097, dtype=torch.float64)  # domain volume: Simpson's rule on r^3
        V3 = _radius(c["alpha"], torch.tensor(c["x1_out"], dtype=torch.float64), x2) ** 3 - \
            _radius(c["alpha"], torch.tensor(-1.0, dtype=torch.float64), x2) ** 3
        w = torch.ones(4097, dtype=torch.float64)
        w[1:-1:2], w[2:-1:2] = 4.0, 2.0
        vol = float((w * V3).sum()) * (2.0 / 4096 / 3.0) * 2.0 * math.pi / 3.0
        rho = vol / c["n"] * (_weigh(c, st[1][:, 0], st[1][:, 1]) - _weigh(c, st[0][:, 0], st[0][:, 1]))
        rho = rho / _hat_volumes(c, "cuda")
        phi = _field(c, rho)
        h1, h2 = (c["x1_out"] + 1.0) / c["n1"], 2.0 / c["n2"]
        G1, G2 = _slope(phi, h1, 0), _slope(phi, h2, 1)
        return dict(phi=phi, rho=rho, electrons=_rows(c, _moved(c, G1, G2, -1.0, 1.0, st[0]).cpu().numpy()),
                    ions=_rows(c, _moved(c, G1, G2, 1.0, 1836.0, st[1]).cpu().numpy()))
    return None
