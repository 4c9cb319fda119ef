"""The work a user of this library has it do, as a dozen measurable cases.

Each case is a dict of plain values; ``prepare`` builds what a program holds before the call (a
stepped context, a field, buffers), ``run`` makes one pass through the public entry points and
returns what the pass computed, ``work`` says what the pass cannot do without, and ``exact`` states
the same results in 64 bits, from the method's equations written out in plain torch.

The kinds of case:
  steps     n steps of one lattice or a batch, then the stored state of every lattice read back to a
            device buffer; optionally one sampling period (fields, spectra, pressure) inside it, the
            conserved masses, or the spectrum and pressure a short run ends with
  slab      one window of a lattice cut into x-slabs: single steps, the boundary columns exported and
            the halo columns imported after each
  spectra   seeds of one configuration, sampled every few steps with correlations on, and the
            averages read to the host
  gradient  the mean-pressure shift and its gradient by the reverse sweep
  snapshot  the power spectrum of one field
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1808_05168_gb300 import LatticeParams, Simulation, capi, workloads

C_X = (0, 1, 0, -1, 0, 1, -1, -1, 1)
C_Z = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
NORM = (1.0, 1 / 3, 1 / 3, 4.0, 4 / 9, 1 / 9, 2 / 3, 2 / 3, 16.0)  # Table I

UNIT_RATES = {"lambda_s": 1.0, "lambda_d": 0.8, "lambda_e": 1.0, "lambda_q": 1.0, "lambda_eps": 1.0}
GENERAL_RATES = {"lambda_s": 1.2, "lambda_d": 0.9, "lambda_e": 1.1, "lambda_q": 1.3, "lambda_eps": 0.95}

# Arithmetic of one lattice update, in operations: densities, moments, forces, collision and the
# inverse transform of both species (350), seven Box-Muller pairs (about 25 each); the integer work
# of the four Philox calls is not counted.
FLOPS_PER_UPDATE = 525
# The transposed step recomputes the forward quantities and applies the transposed Jacobian.
FLOPS_PER_ADJOINT = 900


# ---------------------------------------------------------------------------------- the cases
def _steps(name, Lx, Lz, steps, precision, **kw):
    c = {"name": name, "kind": "steps", "Lx": Lx, "Lz": Lz, "n": 1, "seeds": 0, "steps": steps, "precision": precision,
         "kT": 1e-5, "G": 0.5, "dc": 0.5, "unit_rates": True, "astar": True, "wall_fixed": False, "noise_loc": False,
         "persistent": True, "sample": False, "read": False, "mass": False}
    c.update(kw)
    return c


def listed():
    return [
        # The paper's smallest check of the method (ideal mixture, plain FP64): a hundred steps of one
        # small lattice with its sample, then S_c(q_x) and the mean pressure.  Launches and latency count.
        _steps("ideal_64x32_fp64", 64, 32, 100, "fp64", G=0.0, sample=True, read=True),
        # One rank of an x-slab run: 512 own columns and two halo columns a side, four single steps with
        # the exchange of boundary columns after each.  The smallest calls, one after the other.
        {"name": "slab_516x256_dev32", "kind": "slab", "Lx": 516, "Lz": 256, "Lx_global": 2048, "x0": 510, "steps": 4,
         "precision": "dev32", "kT": 1e-5, "G": 0.5, "dc": 0.5},
        # The long production run (2e5 steps, every diagnostic sampled every 100): one of its periods, in
        # both storage types.
        _steps("production_512x256_dev32", 512, 256, 100, "dev32", sample=True),
        _steps("production_512x256_fp64", 512, 256, 100, "fp64", sample=True),
        # An odd width with every option the method has: general rates, local noise, fixed wall
        # composition, no diffusion correction, plain launches, and the masses watched.
        _steps("odd_641x187_dev32", 641, 187, 40, "dev32", unit_rates=False, astar=False, wall_fixed=True, noise_loc=True,
               persistent=False, mass=True),
        # The batched ensemble (64 seeds x four wall distances x three gradients, 66.8 M sites): one
        # sampling period, the benchmark's step.
        _steps("ensemble_768_dev32", 0, 0, 100, "dev32", seeds=64, sample=True),
        # The throughput run on one large lattice, in both storage types; in FP32 with the masses, whose
        # drift such a run watches.
        _steps("large_8192x2048_dev32", 8192, 2048, 50, "dev32", mass=True),
        _steps("large_8192x2048_fp64", 8192, 2048, 4, "fp64"),
        # Seed-averaged spectra and correlations at the paper's size (L = 32, Lx = 128) as the protocols
        # measure them: default launches, a sample every ten steps, averages read to the host.
        {"name": "spectra_32x128x32_dev32", "kind": "spectra", "Lx": 128, "Lz": 32, "n": 32, "steps": 400, "every": 10,
         "precision": "dev32", "kT": 1e-4, "G": 0.3, "dc": 0.32},
        # The gradient of the mean-pressure shift on its own configuration, and eight seeds of it in one
        # sweep from FP32 state (kT of the paper's non-equilibrium runs).
        {"name": "gradient_256x128_fp64", "kind": "gradient", "Lx": 256, "Lz": 128, "n": 1, "steps": 500, "ckpt": 100,
         "precision": "fp64", "kT": 1e-4, "G": 0.5, "dc": 0.5, "options": False},
        {"name": "gradient_8x256x128_dev32", "kind": "gradient", "Lx": 256, "Lz": 128, "n": 8, "steps": 300, "ckpt": 100,
         "precision": "dev32", "kT": 1e-4, "G": 0.5, "dc": 0.5, "options": False},
        # The spectrum of one snapshot of a field.
        {"name": "snapshot_2048x1024", "kind": "snapshot", "Lx": 2048, "Lz": 1024, "noalloc": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: its kind, then sizes spread over the logarithm of their range."""
    kind = rng.choice(["steps", "steps", "steps", "period", "slab", "spectra", "gradient", "snapshot"])
    precision = rng.choice(["dev32", "dev32", "fp64"])
    dc = rng.choice([0.1, 0.3, 0.5])
    if kind == "steps":
        Lx, Lz = _log_int(rng, 24, 6000), _log_int(rng, 12, 1500)
        most = 1 << (25 if precision == "dev32" else 21)  # sites
        while Lx * Lz > most:
            Lx, Lz = (Lx + 1) // 2 + 1, (Lz + 1) // 2 + 1
        n = max(1, min(_log_int(rng, 1, 48), most // (Lx * Lz)))
        updates = 6e8 if precision == "dev32" else 2.5e7
        steps = int(max(1, min(_log_int(rng, 1, 200), updates // (n * Lx * Lz))))
        c = _steps("", Lx, Lz, steps, precision, n=n, dc=dc, kT=rng.choice([1e-6, 1e-5, 1e-4]), G=rng.choice([0.0, 0.3, 0.5]),
                   unit_rates=rng.random() < 0.6, astar=rng.random() < 0.8, wall_fixed=rng.random() < 0.25,
                   noise_loc=rng.random() < 0.25, persistent=rng.random() < 0.6, mass=rng.random() < 0.3)
    elif kind == "period":
        Lx, Lz = 1 << rng.randint(6, 11), 1 << rng.randint(5, 10)
        most = 1 << (21 if precision == "dev32" else 17)
        n = max(1, min(_log_int(rng, 1, 32), most // (Lx * Lz)))
        while Lx * Lz > most:
            Lx //= 2
        c = _steps("", Lx, Lz, _log_int(rng, 10, 100), precision, n=n, dc=dc, sample=True, read=rng.random() < 0.5,
                   persistent=rng.random() < 0.7)
    elif kind == "slab":
        own, Lz = 2 * _log_int(rng, 16, 2048), _log_int(rng, 16, 700)
        c = {"kind": "slab", "Lx": own + 4, "Lz": Lz, "Lx_global": 4 * own, "x0": own - 2, "steps": rng.randint(1, 8),
             "precision": precision, "kT": 1e-5, "G": 0.5, "dc": dc}
    elif kind == "spectra":
        Lz = rng.choice([16, 32, 64])
        c = {"kind": "spectra", "Lx": Lz * rng.choice([2, 4]), "Lz": Lz, "n": _log_int(rng, 2, 32 * 32 // Lz),
             "steps": 10 * _log_int(rng, 2, 40), "every": rng.choice([5, 10]), "precision": precision, "kT": 1e-4, "G": 0.3, "dc": dc}
        if precision == "fp64":
            c["n"], c["steps"] = min(c["n"], 8), min(c["steps"], 100)
    elif kind == "gradient":
        Lx, Lz = _log_int(rng, 32, 320), _log_int(rng, 16, 160)
        c = {"kind": "gradient", "Lx": Lx, "Lz": Lz, "n": rng.choice([1, 1, 2, 4]), "steps": _log_int(rng, 60, 400),
             "ckpt": rng.choice([20, 50]), "precision": precision, "kT": 1e-4, "G": rng.choice([0.3, 0.5]), "dc": dc,
             "options": rng.random() < 0.3}
    else:
        Lx, Lz = 1 << rng.randint(5, 12), 1 << rng.randint(4, 12)
        while Lx * Lz > 1 << 23:
            Lx //= 2
        c = {"kind": "snapshot", "Lx": Lx, "Lz": Lz, "noalloc": Lx * Lz <= capi.LB_NOALLOC_MAX_POINTS and rng.random() < 0.5}
    c.pop("name", None)
    return c


# ------------------------------------------------------------------------------ what the cases use
def _lattices(case, seed):
    """The lattices of a case; their noise is keyed by the seed."""
    key = 1000 + 7919 * (seed % 100003)
    if case.get("seeds"):
        return workloads.c3(n_seeds=case["seeds"], seed0=key)
    rates = UNIT_RATES if case.get("unit_rates", True) else GENERAL_RATES
    n = case.get("n", 1)
    return [LatticeParams(case["Lx"], case["Lz"], kT=case["kT"], G=case["G"], grad_c0=case["dc"] / case["Lz"], seed=key + i,
                          lattice_id=i, **rates) for i in range(n)]


def _groups(lattices):
    """Indices of the lattices by shape, so that equal ones are handled together."""
    by = {}
    for i, p in enumerate(lattices):
        by.setdefault((p.Lx, p.Lz), []).append(i)
    return by


def _c0(p, device="cuda"):
    z = torch.arange(p.Lz, dtype=torch.float64, device=device) + 0.5 - 0.5 * p.Lz
    return 0.5 + z * p.grad_c0


def _background(p):
    """w_l rho_bar c^S_0(z): [2, 9, Lz, 1]."""
    c = _c0(p)
    w = torch.tensor(W, dtype=torch.float64, device="cuda").view(9, 1)
    return torch.stack([w * c, w * (1 - c)]).unsqueeze(-1)


def _initial(lattices, precision, seed):
    """A thermal state for every lattice, in the storage type and the layout of import_columns
    ([18][Lz][Lx]): independent fluctuations of variance w_l kT / 2 about the background (about what
    a long run has), those of lattices of one shape drawn together."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    sd = torch.tensor([math.sqrt(w / 2) for w in W], device="cuda").repeat(2).view(18, 1, 1)
    out = [None] * len(lattices)
    for (Lx, Lz), idx in _groups(lattices).items():
        for first in range(0, len(idx), 32):
            part = idx[first:first + 32]
            x = torch.randn((len(part), 18, Lz, Lx), generator=g, device="cuda") * sd
            for k, i in enumerate(part):
                p = lattices[i]
                d = x[k] * math.sqrt(p.kT if p.kT > 0 else 1e-5)
                if precision == "fp64":
                    d = d.double() + _background(p).reshape(18, Lz, 1)
                out[i] = d.contiguous()
    return out


def _read_state(sim, views):
    for i, v in enumerate(views):
        sim.export_columns(0, v.shape[2], out=v, lattice=i)


def _views(lattices, flat):
    v, at = [], 0
    for p in lattices:
        n = 18 * p.Lz * p.Lx
        v.append(flat[at:at + n].view(18, p.Lz, p.Lx))
        at += n
    return v


def _storage(precision):
    return torch.float32 if precision == "dev32" else torch.float64


class State:
    """What a program keeps between passes."""


def prepare(case, seed):
    s = State()
    s.case = case
    kind = case["kind"]
    s.stream = torch.cuda.Stream()
    if kind == "snapshot":
        g = torch.Generator(device="cuda")
        g.manual_seed(int(seed))
        s.field = torch.randn((case["Lz"], case["Lx"]), generator=g, dtype=torch.float64, device="cuda") * 1e-3
        s.out = torch.empty_like(s.field)
        s.call = capi.lb_power_spectrum_noalloc if case["noalloc"] else capi.lb_power_spectrum
        torch.cuda.synchronize()
        return s
    s.lattices = lattices = _lattices(case, seed)
    if kind == "gradient":
        options = {"astar": False, "wall_fixed": True, "noise_loc": True} if case["options"] else {}
        s.sim = Simulation(lattices, precision=case["precision"], **options)
        return s
    if kind == "steps":
        fast = case["persistent"]
        s.sim = Simulation(lattices, precision=case["precision"], astar=case["astar"], wall_fixed=case["wall_fixed"],
                           noise_loc=case["noise_loc"], graph=fast, persistent=fast, autotune=fast)
        every = case["steps"] if case["sample"] else 0
    elif kind == "slab":
        s.sim = Simulation(lattices, precision=case["precision"])
        s.sim.set_site_map(case["x0"], case["Lx_global"])
        every = 0
    else:
        s.sim = Simulation(lattices, precision=case["precision"])
        every = case["every"]
    s.sim.set_stream(s.stream)
    if every:
        s.sim.set_sampling(0, every)
    if kind == "spectra":
        s.sim.set_correlations(("c", "ux"), modes=(1, 2))
    # the run is under way (the tile is chosen, graphs are captured): a pass's worth of steps, then
    # the state of this seed
    s.sim.step(case["steps"])
    s.sim.synchronize()
    init = _initial(lattices, case["precision"], seed)
    torch.cuda.synchronize()
    for i, d in enumerate(init):
        s.sim.import_columns(0, d, lattice=i)
    s.sim.synchronize()
    if every:
        s.sim.reset_statistics()
    sites = sum(p.Lx * p.Lz for p in lattices)
    dtype = _storage(case["precision"])
    if kind in ("steps", "slab"):
        s.out = torch.empty(18 * sites, dtype=dtype, device="cuda")
        s.views = _views(lattices, s.out)
    if kind == "slab":
        s.halos = _halos(case, seed)
        s.sent = [[torch.empty((18, case["Lz"], 2), dtype=dtype, device="cuda") for _ in range(2)] for _ in range(case["steps"])]
        torch.cuda.synchronize()
    return s


def _halos(case, seed):
    """What the neighbours send after each step: columns of their thermal state."""
    p = LatticeParams(4 * case["steps"], case["Lz"], kT=case["kT"], grad_c0=case["dc"] / case["Lz"])
    x = _initial([p], case["precision"], seed + 1000003)[0]
    return [[x[:, :, 4 * k:4 * k + 2].contiguous(), x[:, :, 4 * k + 2:4 * k + 4].contiguous()] for k in range(case["steps"])]


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "snapshot":
        s.call(s.field.data_ptr(), case["Lx"], case["Lz"], s.out.data_ptr(), s.stream.cuda_stream)
        return s.out
    sim = s.sim
    if kind == "gradient":
        losses, grads = sim.pressure_shift_gradients(case["steps"], case["ckpt"])
        return {"loss": losses, "grad": grads}
    if kind == "steps":
        sim.step(case["steps"])
        _read_state(sim, s.views)
        out = {"state": s.out}
        if case["read"]:
            out["S_c"] = np.stack([sim.structure_factor("c", lattice=i, qz0_only=True)[0] for i in range(len(s.lattices))])
            out["pressure"] = np.array([sim.mean_pressure(i) for i in range(len(s.lattices))])
        if case["mass"]:
            out["mass"] = np.stack([sim.mass(i) for i in range(len(s.lattices))])
        return out
    if kind == "slab":
        Lx = case["Lx"]
        for k in range(case["steps"]):
            sim.step(1)
            sim.export_columns(2, 2, out=s.sent[k][0])
            sim.export_columns(Lx - 4, 2, out=s.sent[k][1])
            sim.import_columns(0, s.halos[k][0])
            sim.import_columns(Lx - 2, s.halos[k][1])
        _read_state(sim, s.views)
        return {"state": s.out, "sent": s.sent}
    sim.step(case["steps"])
    n = range(len(s.lattices))
    return {"S_c": np.stack([sim.structure_factor("c", lattice=i)[0] for i in n]),
            "S_ux": np.stack([sim.structure_factor("ux", lattice=i)[0] for i in n]),
            "R_c": np.stack([sim.correlation("c", lattice=i)[0] for i in n]),
            "R_ux": np.stack([sim.correlation("ux", lattice=i)[0] for i in n]),
            "C_c": np.stack([sim.mode_correlation("c", 0, lattice=i)[0] for i in n]),
            "rho": np.stack([sim.profile("rho", lattice=i)[0] for i in n]),
            "p": np.stack([sim.profile("p", lattice=i)[0] for i in n]),
            "pressure": np.array([sim.mean_pressure(i) for i in n])}


def work(case):
    """Bytes: the state (or field) read once and written once, what is handed out written once.
    Operations: the updates of the pass."""
    kind = case["kind"]
    if kind == "snapshot":
        n = case["Lx"] * case["Lz"]
        return {"bytes": 16.0 * n, "flops": 2.5 * n * math.log2(n) + 3 * n}
    sites = sum(p.Lx * p.Lz for p in _lattices(case, 0))
    real = 4 if case["precision"] == "dev32" else 8
    updates = float(case["steps"]) * sites
    if kind == "gradient":
        # two runs (with and without noise); the one without is the same in every column
        return {"bytes": 2.0 * 18 * real * sites, "flops": updates * (FLOPS_PER_UPDATE + FLOPS_PER_ADJOINT)}
    state = 18.0 * real * sites
    if kind in ("steps", "slab"):
        return {"bytes": 3 * state, "flops": updates * FLOPS_PER_UPDATE}
    samples = case["steps"] / case["every"]
    p = _lattices(case, 0)[0]
    fft = 2.5 * 4 * math.log2(p.Lx * p.Lz)
    return {"bytes": 2 * state + 8.0 * sites * 4, "flops": updates * FLOPS_PER_UPDATE + samples * sites * (fft + 2 * 2 * p.Lz)}


# ------------------------------------------------------------- the method in 64 bits, plain torch
def _hi_lo(m, x):
    p = m * x  # 64-bit products wrap; the halves are exact
    return (p >> 32) & 0xFFFFFFFF, p & 0xFFFFFFFF


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    x = [c0, c1, c2, c3]
    for r in range(10):
        a, b = (k0 + r * 0x9E3779B9) & 0xFFFFFFFF, (k1 + r * 0xBB67AE85) & 0xFFFFFFFF
        h0, l0 = _hi_lo(0xD2511F53, x[0])
        h1, l1 = _hi_lo(0xCD9E8D57, x[2])
        x = [h1 ^ x[1] ^ a, l1, h0 ^ x[3] ^ b, l0]
    return x


def _normals(site, step, lid, key):
    """The fourteen normals of every site; site [Lz, Lx], lid and key [B]."""
    B = len(lid)
    lid = torch.tensor(lid, dtype=torch.int64, device="cuda").view(B, 1, 1)
    k0 = torch.tensor([k & 0xFFFFFFFF for k in key], dtype=torch.int64, device="cuda").view(B, 1, 1)
    k1 = torch.tensor([k >> 32 for k in key], dtype=torch.int64, device="cuda").view(B, 1, 1)
    c0 = site.unsqueeze(0).expand(B, -1, -1)
    out = []
    for call in range(4):
        w = _philox(c0, torch.full_like(c0, step), lid.expand_as(c0), torch.full_like(c0, call), k0, k1)
        for a, b in ((w[0], w[1]), (w[2], w[3]))[: 2 if call < 3 else 1]:
            u1 = (2 * (a & 0x7FFFFF) + 1).double() * 2.0 ** -24
            u2 = (2 * (b & 0x7FFFFF) + 1).double() * 2.0 ** -24
            r = torch.sqrt(-2 * torch.log(u1))
            out += [r * torch.cos(2 * math.pi * u2), r * torch.sin(2 * math.pi * u2)]
    return out


class Method:
    """The step of lattices of one shape, populations [B, 2, 9, Lz, Lx] in double precision."""

    def __init__(self, lattices, astar=True, wall_fixed=False, noise_loc=False, x0=0, Lx_global=None, grad=False):
        p0 = lattices[0]
        self.p, self.B, self.Lx, self.Lz = lattices, len(lattices), p0.Lx, p0.Lz
        self.astar, self.wall_fixed, self.noise_loc = astar, wall_fixed, noise_loc
        t = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda").view(self.B, 1, 1)  # noqa: E731
        self.G, self.ls, self.ld = (t([getattr(p, k) for p in lattices]) for k in ("G", "lambda_s", "lambda_d"))
        if grad:
            for v in (self.G, self.ls, self.ld):
                v.requires_grad_()
        self.le = t([p.lambda_s if p.lambda_e is None else p.lambda_e for p in lattices])
        self.lq, self.leps = t([p.lambda_q for p in lattices]), t([p.lambda_eps for p in lattices])
        self.kT, self.g3 = t([p.kT for p in lattices]), t([p.grad_c0 / 3 for p in lattices])
        self.c0 = torch.stack([_c0(p) for p in lattices]).unsqueeze(-1)
        self.cw = [t([0.5 + s * 0.5 * p.Lz * p.grad_c0 for p in lattices]) for s in (-1, 1)]
        Lg = Lx_global or self.Lx
        z = torch.arange(self.Lz, dtype=torch.int64, device="cuda").view(-1, 1)
        x = torch.arange(self.Lx, dtype=torch.int64, device="cuda").view(1, -1)
        self.site = z * Lg + (x + x0) % Lg
        self.noisy = any(p.kT > 0 for p in lattices)

    def rest(self):
        return torch.stack([_background(p).expand(2, 9, p.Lz, p.Lx) for p in self.p]).clone()

    def pull(self, f):
        v = []
        for l in range(9):
            g = torch.roll(f[:, :, l], C_X[l], dims=-1) if C_X[l] else f[:, :, l]
            if C_Z[l] > 0:
                g = torch.cat([f[:, :, OPP[l], :1], g[:, :, :-1]], dim=2)
            elif C_Z[l] < 0:
                g = torch.cat([g[:, :, 1:], f[:, :, OPP[l], -1:]], dim=2)
            v.append(g)
        return v

    def moments(self, v):
        a57, a68, d13, d24 = v[5] - v[7], v[6] - v[8], v[1] - v[3], v[2] - v[4]
        s13, s24, s57, s68 = v[1] + v[3], v[2] + v[4], v[5] + v[7], v[6] + v[8]
        e, dg = s13 + s24, s57 + s68
        return [v[0] + e + dg, d13 + a57 - a68, d24 + a57 + a68, -2 * v[0] + e + 4 * dg, s13 - s24, s57 - s68,
                -d13 + 2 * (a57 - a68), -d24 + 2 * (a57 + a68), 2 * v[0] - 4 * e + 8 * dg]

    def neighbours(self, rho):
        """sum_l w_l c_l rho(r + c_l) (x, z) and sum_l w_l |c_l|^2 rho(r + c_l), wall ghosts included."""
        ends = []
        for row, cw in ((rho[:, :, :1], self.cw[0]), (rho[:, :, -1:], self.cw[1])):
            if self.wall_fixed:
                tot = row.sum(dim=1)
                row = torch.stack([tot * cw, tot * (1 - cw)], dim=1)
            ends.append(row)
        r = torch.cat([ends[0], rho, ends[1]], dim=2)
        up, mid, dn = r[:, :, 2:], r[:, :, 1:-1], r[:, :, :-2]
        e = lambda a: torch.roll(a, -1, dims=-1)  # noqa: E731
        w = lambda a: torch.roll(a, 1, dims=-1)  # noqa: E731
        ne, nw, se, sw = e(up), w(up), e(dn), w(dn)
        sx = (e(mid) - w(mid)) / 9 + (ne - nw + se - sw) / 36
        sz = (up - dn) / 9 + (ne + nw - se - sw) / 36
        N = (e(mid) + w(mid) + up + dn) / 9 + (ne + nw + se + sw) / 18
        return sx, sz, N

    def step(self, f, t, sample=False):
        """f after one step; with sample also (fields [B, 4, Lz, Lx], pressure [B, Lz, Lx])."""
        m = self.moments(self.pull(f))
        rs = m[0]
        rho = rs.sum(dim=1)
        sx, sz, N = self.neighbours(rs)
        A, Bs = 0, 1
        FA = [-self.G * rs[:, A] * s[:, Bs] for s in (sx, sz)]
        FB = [-self.G * rs[:, Bs] * s[:, A] for s in (sx, sz)]
        FN = [FA[0] + FB[0], FA[1] + FB[1]]
        if self.astar:
            F = [torch.stack([rs[:, A] / rho * FN[k], rs[:, Bs] / rho * FN[k]], dim=1) for k in (0, 1)]
        else:
            F = [torch.stack([FA[k], FB[k]], dim=1) for k in (0, 1)]
        F[1] = F[1] + torch.stack([rho * self.g3, -rho * self.g3], dim=1)
        U = [((m[1 + k].sum(dim=1) + 0.5 * FN[k]) / rho).unsqueeze(1) for k in (0, 1)]
        ux, uz = U
        lam = [None, self.ld, self.ld, self.le, self.ls, self.ls, self.lq, self.lq, self.leps]
        eq = [rs, rs * ux, rs * uz, 3 * rs * (ux * ux + uz * uz), rs * (ux * ux - uz * uz), rs * ux * uz, 0, 0, 0]
        src = [0, F[0], F[1], 6 * (ux * F[0] + uz * F[1]), 2 * (ux * F[0] - uz * F[1]), ux * F[1] + uz * F[0], 0, 0, 0]
        n = _normals(self.site, t, [p.lattice_id for p in self.p], [p.seed for p in self.p]) if self.noisy else None
        ms = [rs]
        for a in range(1, 9):
            L = lam[a].unsqueeze(1)
            v = (1 - L) * m[a] + L * eq[a] + (1 - 0.5 * L) * src[a]
            if self.noisy:
                if a <= 2:
                    red = rs[:, A] * rs[:, Bs] / rho if self.noise_loc else 0.25
                    xi = torch.sqrt((2 - lam[a]) * lam[a] * self.kT * red) * n[a - 1]
                    v = v + torch.stack([xi, -xi], dim=1)
                else:
                    ref = rs if self.noise_loc else 0.5
                    v = v + torch.sqrt(3 * (2 - L) * L * NORM[a] * self.kT.unsqueeze(1) * ref) * torch.stack([n[a - 1], n[a + 5]], dim=1)
            ms.append(v)
        q = [ms[a] / NORM[a] for a in range(9)]
        b4, b5 = q[0] + q[3] - 4 * q[8], q[0] + 4 * q[3] + 8 * q[8]
        g = [q[0] - 2 * q[3] + 2 * q[8], b4 + q[1] + q[4] - q[6], b4 + q[2] - q[4] - q[7], b4 - q[1] + q[4] + q[6],
             b4 - q[2] - q[4] + q[7], b5 + q[1] + q[2] + q[5] + 2 * q[6] + 2 * q[7], b5 - q[1] + q[2] - q[5] - 2 * q[6] + 2 * q[7],
             b5 - q[1] - q[2] + q[5] - 2 * q[6] - 2 * q[7], b5 + q[1] - q[2] - q[5] + 2 * q[6] - 2 * q[7]]
        out = torch.stack([W[l] * g[l] for l in range(9)], dim=2)
        if not sample:
            return out
        P = (m[3] + 2 * m[0]).sum(dim=1) / 6 + 0.25 * self.G * (rs[:, A] * N[:, Bs] + rs[:, Bs] * N[:, A])
        fields = torch.stack([rho - 1, rs[:, A] / rho - self.c0, ux.squeeze(1), uz.squeeze(1)], dim=1)
        return out, fields, P


def exact(case, seed):
    kind = case["kind"]
    if kind == "snapshot":
        s = prepare(case, seed)
        return torch.fft.fft2(s.field).abs().square() / (case["Lx"] * case["Lz"])
    lattices = _lattices(case, seed)
    updates = float(case["steps"]) * sum(p.Lx * p.Lz for p in lattices)
    if kind == "gradient":
        if updates > 9e7 or case["steps"] > 600:
            return None  # over 20 seconds
        return _exact_gradient(case, lattices)
    if updates > 1.2e9 or len(_groups(lattices)) > 1:
        return None
    opts = {k: case[k] for k in ("astar", "wall_fixed", "noise_loc") if k in case}
    if kind == "slab":
        opts.update(x0=case["x0"], Lx_global=case["Lx_global"])
    p0 = lattices[0]
    init = _initial(lattices, case["precision"], seed)
    f = torch.stack(init).double().view(len(lattices), 2, 9, p0.Lz, p0.Lx)
    bg = torch.stack([_background(p) for p in lattices])
    if case["precision"] == "dev32":
        f = f + bg
    M = Method(lattices, **opts)
    del init
    every = case["every"] if kind == "spectra" else (case["steps"] if kind == "steps" and case["sample"] else 0)
    halos = _halos(case, seed) if kind == "slab" else None
    stored = lambda a: a - bg if case["precision"] == "dev32" else a  # noqa: E731
    sums, count, sent = {}, 0, []
    for k in range(case["steps"]):
        t = case["steps"] + k  # prepare() has taken as many steps before
        if every and t % every == 0:
            f, fields, P = M.step(f, t, sample=True)
            count += 1
            add = {"S": torch.fft.fft2(fields).abs().square() / (p0.Lx * p0.Lz), "P": P.mean(dim=(1, 2)), "p": P.mean(dim=2),
                   "rho": fields[:, 0].mean(dim=2) + 1, "R": torch.einsum("bfzx,bfyx->bfzy", fields, fields) / p0.Lx}
            if kind == "spectra":
                X = torch.fft.fft(fields[:, 1], dim=-1)[..., 1]
                add["C"] = X.conj().unsqueeze(2) * X.unsqueeze(1) / p0.Lx
            last = add["P"]
            for key, v in add.items():
                sums[key] = sums[key] + v if key in sums else v
        else:
            f = M.step(f, t)
        if kind == "slab":
            now = stored(f).reshape(18, p0.Lz, p0.Lx)
            sent.append([now[:, :, 2:4].clone(), now[:, :, -4:-2].clone()])
            b = bg.reshape(18, p0.Lz, 1) if case["precision"] == "dev32" else 0
            flat = f.view(18, p0.Lz, p0.Lx)
            flat[:, :, :2] = halos[k][0].double() + b
            flat[:, :, -2:] = halos[k][1].double() + b
    mean = {key: v / count for key, v in sums.items()}
    if kind == "spectra":
        return {"S_c": mean["S"][:, 1], "S_ux": mean["S"][:, 2], "R_c": mean["R"][:, 1], "R_ux": mean["R"][:, 2],
                "C_c": mean["C"], "rho": mean["rho"], "p": mean["p"], "pressure": torch.stack([last, mean["P"]], dim=1)}
    out = {"state": stored(f).reshape(-1)}
    if kind == "slab":
        out["sent"] = sent
        return out
    if case["read"]:
        out["S_c"] = mean["S"][:, 1, 0, :]
        out["pressure"] = torch.stack([last, mean["P"]], dim=1)
    if case["mass"]:
        out["mass"] = f.sum(dim=(2, 3, 4))
    return out


def _exact_gradient(case, lattices):
    """Loss and gradient of the mean-pressure shift: the forward states of each run kept, then every
    step differentiated by torch's reverse mode, last to first."""
    opts = {"astar": False, "wall_fixed": True, "noise_loc": True} if case["options"] else {}
    T, sites = case["steps"], lattices[0].Lx * lattices[0].Lz
    loss, grad = 0, 0
    for sign in (1.0, -1.0):
        run = lattices if sign > 0 else [LatticeParams(**{**vars(p), "kT": 0.0}) for p in lattices]
        M = Method(run, grad=True, **opts)
        with torch.no_grad():
            states, total = [M.rest()], 0
            for t in range(T):
                f, _, P = M.step(states[-1], t, sample=True)
                total = total + P.mean(dim=(1, 2))
                states.append(f)
        loss = loss + sign * total / T
        bar = torch.zeros_like(states[0])
        states.pop()
        for t in reversed(range(T)):
            f = states.pop().requires_grad_()
            g, _, P = M.step(f, t, sample=True)
            obj = (g * bar).sum() + sign * P.sum() / (T * sites)
            bar, dG, ds, dd = torch.autograd.grad(obj, [f, M.G, M.ls, M.ld])
            grad = grad + torch.stack([dG.view(-1), ds.view(-1), dd.view(-1)], dim=1)
    return {"loss": loss, "grad": grad}
