"""Timed cases of the framework's main path: what a user's program has it do through its public
entry points, from the smallest workload to the largest.

A case is a dict of plain values. ``prepare`` makes what the program holds before the call,
``run`` is one pass, ``work`` the bytes and operations the pass cannot do without, ``exact``
the same outputs in 64 bits by plain numpy where that is possible.

Kinds:

* ``macro``: one projective macro step from a given coarse state (set the state, lift, burst
  with the restriction samples, project, read the new state), the call a production run
  repeats. Every coarse variable, both boundaries, both electron models.
* ``pic``: 20 resolved PIC steps and a measurement of the coarse state, as the resolved
  reference runs do (particles sorted every 20 steps).
* ``ensemble``: one macro step of a batch of realisations of mixed sizes and boundaries.
* ``field``: one field solve from the previous step's potential (a time loop of the caller's own).
* ``restrict``: deposit, restriction sample and coarsening of particles the caller holds, in no
  velocity order (any layout a caller's own loader produces) and of any count.
* ``diag``: conserved quantities of a particle state.
* ``train`` / ``infer``: the surrogate network's training steps and its evaluation.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1610_01071_gb300 as pe

DEV = "cuda"


def listed():
    iaw, slab, kin = (pe.inputs.workload(k) for k in ("iaw_large", "slab", "iaw_kinetic"))
    small = pe.inputs.workload("iaw_small")
    return [
        # the smallest workload: a macro step of 128 cells is a chain of short launches
        _macro("macro_small", small["ncell"], small["N"] // small["ncell"], small["K"], small["M"],
               small["n_coarse"]),
        # the benchmark's workload
        _macro("macro_large", iaw["ncell"], iaw["N"] // iaw["ncell"], iaw["K"], iaw["M"], iaw["n_coarse"]),
        # the largest: the slab expansion between absorbing walls with the phase-space variable
        _macro("macro_slab_phase", slab["ncell"], slab["N"] // slab["ncell"], 15, 4, slab["n_coarse"],
               coarse="phase_space", n_v=64, boundary="absorbing"),
        # the paper's phase-space variable as it states it (coiflets along v), a particle count per
        # cell that is no power of two
        _macro("macro_wavelet_odd", 1024, 1500, 20, 5, 64, coarse="phase_space", n_v=256, n_v_coarse=64,
               wavelet="coif4"),
        # resolved runs: one species with an odd count per cell, and the two-species workload
        _pic("pic_odd", 2048, 1237),
        _pic("pic_kinetic", kin["ncell"], kin["N"] // kin["ncell"], electrons="kinetic"),
        # many realisations at once: parameter studies and the surrogate's training data
        dict(name="ensemble", kind="ensemble", members=24, mix=4, log2cells_lo=9, log2cells_hi=13, log2n_lo=18,
             log2n_hi=21, K=20, M=10),
        # a caller's own time loop around single kernels
        dict(name="field_periodic", kind="field", ncell=4096, dx=0.5, boundary="periodic", mode="boltzmann"),
        dict(name="restrict_odd", kind="restrict", ncell=1024, N=3000001, n_coarse=64, wavelet="haar", tau=4.0),
        dict(name="diag_large", kind="diag", ncell=4096, N=1 << 23),
        # the surrogate: training on the coarse slopes of an ensemble, and the one evaluation of a
        # gated macro step
        dict(name="train", kind="train", d=512, hidden=512, layers=4, B=2048, nsteps=20, pairs=8192),
        dict(name="infer_one", kind="infer", d=512, hidden=512, layers=4, B=1, f64=True),
    ]


def _macro(name, ncell, ppc, K, M, n_coarse, coarse="moments", n_v=64, n_v_coarse=0, wavelet="haar",
           boundary="periodic", electrons="boltzmann"):
    return dict(name=name, kind="macro", ncell=int(ncell), ppc=int(ppc), K=int(K), M=int(M), n_coarse=int(n_coarse),
                coarse=coarse, n_v=int(n_v), n_v_coarse=int(n_v_coarse), wavelet=wavelet, boundary=boundary,
                electrons=electrons)


def _pic(name, ncell, ppc, boundary="periodic", electrons="boltzmann"):
    return dict(name=name, kind="pic", ncell=int(ncell), ppc=int(ppc), boundary=boundary, electrons=electrons)


def _log2(rng, lo, hi):
    return int(round(2.0 ** rng.uniform(math.log2(lo), math.log2(hi))))


def draw(rng):
    kind = rng.choice(["macro", "macro", "macro", "macro", "pic", "pic", "ensemble", "field", "restrict", "diag",
                       "train", "infer"])
    if kind in ("macro", "pic"):
        ncell = 1 << rng.randint(7, 13)
        # particles per cell: powers of two (the quiet start's ordered storage) and any other count
        ppc = 1 << rng.randint(6, 12) if rng.random() < 0.5 else _log2(rng, 64, 4096)
        ppc = max(32, min(ppc, (1 << 24) // ncell))
        if kind == "pic":
            which = rng.choice(["boltzmann", "boltzmann", "kinetic", "walls"])
            if which == "kinetic":
                ppc = max(32, min(ppc, (1 << 23) // ncell))
            c = _pic("", ncell, ppc, "absorbing" if which == "walls" else "periodic",
                     "kinetic" if which == "kinetic" else "boltzmann")
        else:
            K, M = rng.randint(8, 24), rng.randint(2, 10)
            nc = max(8, ncell >> rng.randint(3, 5))
            var = rng.choice(["moments", "moments", "moments_d4", "pressure", "phase", "wavelet", "kinetic"])
            kw = {}
            if var == "moments_d4":
                kw = dict(wavelet="d4")
            elif var == "pressure":
                kw = dict(coarse="moments_pressure")
                ncell, nc = min(ncell, 4096), min(nc, 512)
            elif var == "phase":
                kw = dict(coarse="phase_space", n_v=rng.choice([32, 64, 100, 128]))
            elif var == "wavelet":
                kw = dict(coarse="phase_space", n_v=rng.choice([128, 256]), n_v_coarse=rng.choice([32, 64]),
                          wavelet=rng.choice(["haar", "coif4"]))
            elif var == "kinetic":
                kw = dict(coarse="phase_space", n_v=64, electrons="kinetic")
                ppc = max(32, min(ppc, (1 << 23) // ncell))
            if var in ("moments", "phase") and rng.random() < 0.4:
                kw["boundary"] = "absorbing"
            c = _macro("", ncell, ppc, K, M, nc, **kw)
        del c["name"]
        return c
    if kind == "ensemble":
        lo = rng.randint(17, 19)
        c = dict(kind=kind, members=rng.randint(6, 32), mix=rng.randint(0, 9999), log2cells_lo=rng.randint(7, 9),
                 log2cells_hi=rng.randint(10, 13), log2n_lo=lo, log2n_hi=lo + 2, K=rng.randint(8, 20),
                 M=rng.randint(2, 10))
        while work(c)["bytes"] > 1.5e10:
            c["members"] -= 1
        return c
    if kind == "field":
        return dict(kind=kind, ncell=1 << rng.randint(6, 13), dx=round(rng.uniform(0.25, 0.75), 4),
                    boundary=rng.choice(["periodic", "absorbing"]),
                    mode=rng.choice(["boltzmann", "boltzmann", "linearized"]))
    if kind == "restrict":
        ncell = 1 << rng.randint(7, 12)
        return dict(kind=kind, ncell=ncell, N=_log2(rng, 20000, 1 << 23), n_coarse=max(8, ncell >> rng.randint(0, 5)),
                    wavelet=rng.choice(["haar", "haar", "d4"]), tau=round(rng.uniform(0.0, 20.0), 3))
    if kind == "diag":
        return dict(kind=kind, ncell=1 << rng.randint(7, 13), N=_log2(rng, 10000, 1 << 23))
    d, h, layers = 64 * rng.randint(1, 8), 64 * rng.randint(2, 16), rng.randint(2, 5)
    if kind == "train":
        return dict(kind=kind, d=d, hidden=h, layers=layers, B=32 * _log2(rng, 2, 64), nsteps=rng.randint(5, 25),
                    pairs=_log2(rng, 1000, 10000))
    return dict(kind=kind, d=d, hidden=h, layers=layers, B=_log2(rng, 1, 2048), f64=rng.random() < 0.5)


# ------------------------------------------------------------------ contexts


def _config(c, seed):
    """The context of a macro or pic case (the time steps and velocity ranges of the package's workloads)."""
    kin = c["electrons"] == "kinetic"
    dt = 0.25 / math.sqrt(1800.0) if kin else 0.1
    K, M, nc = c.get("K", 20), c.get("M", 10), c.get("n_coarse", max(8, c["ncell"] // 16))
    dx = 0.28125 if kin else 0.5
    return pe.make_config(c["ncell"], nc, K, c["ncell"] * c["ppc"], dx * c["ncell"], dt, M * K * dt,
                          v_th=0.22 if kin else 1.0, wavelet=c.get("wavelet", "haar"), sort_every=20, seed=seed,
                          newton_tol=1e-10, newton_maxit=80, coarse=c.get("coarse", "moments"), n_v=c.get("n_v", 64),
                          v_max=2.5 if kin else 8.0,
                          ps_filter=3 if c.get("coarse") == "phase_space" and not c["n_v_coarse"] else 0,
                          boundary=c["boundary"], electrons=c["electrons"], qm_e=-1800.0 if kin else 0.0,
                          n_v_coarse=c.get("n_v_coarse", 0))


def _loaded(cfg, amplitude, walls):
    ctx = pe.Context(cfg, device=DEV)
    if walls:
        ctx.load_initial(profile="slab")
    else:
        ctx.load_initial(amplitude)
    return ctx


def _members(c):
    """(ncell, N, walls) of an ensemble's realisations, sizes uniform in the logarithm."""
    rng = np.random.default_rng(c["mix"])
    out = []
    for i in range(c["members"]):
        ncell = 1 << int(rng.integers(c["log2cells_lo"], c["log2cells_hi"] + 1))
        n = int(2.0 ** rng.uniform(c["log2n_lo"], c["log2n_hi"]))
        out.append((ncell, ncell * max(32, n // ncell), i % 2 == 1))
    return out


# ------------------------------------------------------------------ inputs of the stateless kinds


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _smooth(ncell, g, amp):
    """A few low Fourier modes on the nodes (FP64)."""
    x = torch.arange(ncell, dtype=torch.float64, device=DEV) / ncell
    f = torch.zeros_like(x)
    a = torch.randn(8, generator=g, dtype=torch.float64, device=DEV)
    for m in range(1, 5):
        f += amp / m * (a[2 * m - 2] * torch.cos(2 * math.pi * m * x) + a[2 * m - 1] * torch.sin(2 * math.pi * m * x))
    return f


def _particles(N, ncell, g):
    """Cell-sorted particles, any order of the velocities inside a cell, weights around ncell / N."""
    cell = torch.randint(0, ncell, (N,), generator=g, device=DEV, dtype=torch.int32).sort().values
    theta = torch.rand(N, generator=g, device=DEV)
    v = torch.randn(N, generator=g, device=DEV)
    w = (0.5 + torch.rand(N, generator=g, device=DEV)) * (ncell / N)
    return cell, theta, v, w


def _shift(cap):
    """Largest s with cap 2^s <= 2^22."""
    return 22 - math.ceil(math.log2(cap))


FIELD_SHIFT = 20


def _density(c, g):
    """Fixed-point densities of two successive steps: a wave with particle noise, or a slab in vacuum."""
    n = c["ncell"]
    if c["boundary"] == "periodic":
        base = 1.0 + _smooth(n, g, 0.2).clamp(-0.8, 3.0)
    else:
        x = torch.arange(n, dtype=torch.float64, device=DEV) / n
        base = torch.sigmoid((0.0625 - (x - 0.5).abs()) * 200.0)
    out = []
    for k in range(2):
        noisy = (base * (1.0 + 0.01 * torch.randn(n, generator=g, dtype=torch.float64, device=DEV))).clamp(min=0.0)
        out.append(torch.round(noisy * 2.0 ** (FIELD_SHIFT + 24)).to(torch.int64))
    return out


def _restrict_inputs(c, seed):
    g = _gen(seed)
    parts = _particles(c["N"], c["ncell"], g)
    return parts, _smooth(c["ncell"], g, 0.1).float(), _smooth(c["ncell"], g, 0.1).float()


def _restrict_shifts(c):
    cap = 2.0 * c["ncell"] / c["N"]
    return _shift(cap), _shift(cap * 32.0)


def _bins(c):
    return int(math.log2(c["ncell"] // c["n_coarse"])) if c["wavelet"] == "haar" else 0


def _dims(c):
    return [c["d"]] + [c["hidden"]] * (c["layers"] - 1) + [c["d"]]


def _pairs(c, n, g):
    """Coarse states and slopes: components of different size around their means."""
    scale = 0.1 + torch.rand(c["d"], generator=g, device=DEV)
    X = torch.randn(n, c["d"], generator=g, device=DEV) * scale + torch.randn(c["d"], generator=g, device=DEV)
    Y = torch.tanh(X.roll(1, 1) - X) * scale
    return X, Y


def _weights(c, g):
    dims, parts = _dims(c), []
    for a, b in zip(dims[:-1], dims[1:]):
        parts.append(torch.randn(b * a, generator=g, device=DEV) / math.sqrt(a))
        parts.append(0.1 * torch.randn(b, generator=g, device=DEV))
    return torch.cat(parts)


# ------------------------------------------------------------------ prepare, run


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = dict(case=c, kind=kind)
    if kind in ("macro", "pic"):
        walls = c["boundary"] == "absorbing"
        ctx = _loaded(_config(c, seed), 0.2 if c["electrons"] == "kinetic" else 0.5, walls)
        if kind == "macro":
            ctx.step()
            s["coarse"] = ctx.get_coarse()
        s["ctx"] = ctx
    elif kind == "ensemble":
        s["ctxs"] = []
        for i, (ncell, N, walls) in enumerate(_members(c)):
            cfg = pe.make_config(ncell, min(256, ncell // 16), c["K"], N, 0.5 * ncell, 0.1, c["M"] * c["K"] * 0.1,
                                 seed=seed + 97 * i, newton_tol=1e-10, newton_maxit=80,
                                 boundary="absorbing" if walls else "periodic")
            s["ctxs"].append(_loaded(cfg, 0.1 + 0.4 * (i / c["members"]), walls))
        s["batch"] = pe.Batch(s["ctxs"])
        s["batch"].tune()
        s["batch"].step()
    elif kind == "field":
        s["rho"] = _density(c, _gen(seed))
        s["phi"] = torch.zeros(c["ncell"], dtype=torch.float64, device=DEV)
        s["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
        s["turn"] = 1  # the first pass solves density 0 from the potential of density 1
        _solve(s, tol=1e-12)
    elif kind == "restrict":
        s["parts"], s["Ef"], s["E0f"] = _restrict_inputs(c, seed)
        s["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
        s["rho"] = torch.empty(c["ncell"], dtype=torch.int64, device=DEV)
        s["sample"] = torch.empty((2, c["ncell"] >> _bins(c)), dtype=torch.int64, device=DEV)
    elif kind == "diag":
        g = _gen(seed)
        s["parts"] = _particles(c["N"], c["ncell"], g)
        s["phi"] = _smooth(c["ncell"], g, 0.2)
        s["E"] = -(s["phi"].roll(-1) - s["phi"].roll(1)) / (2 * 0.5)
        s["Ef"] = s["E"].float()
    else:
        g = _gen(seed)
        s["stream"] = torch.cuda.Stream()
        X, Y = _pairs(c, c["pairs"] if kind == "train" else max(64, c["B"]), g)
        p = _weights(c, g)
        torch.cuda.synchronize()
        s["net"] = net = pe.MLP(_dims(c), max_batch=c["B"], device=DEV, stream=s["stream"])
        net.init(seed)
        net.set_params(p)
        net.fit_norm(X, Y, c["d"] // 2 if kind == "train" else 0)
        s["X"], s["Y"], s["seed"] = X, Y, seed
        if kind == "infer":
            x = X[: c["B"]].contiguous()
            s["x"] = x.double() if c["f64"] else x
    torch.cuda.synchronize()
    return s


def _solve(s, tol=1e-10):
    c = s["case"]
    E, Ef, _ = pe.field(s["rho"][s["turn"]], c["ncell"], c["dx"], FIELD_SHIFT, s["phi"], mode=c["mode"], tol=tol,
                        maxit=200, status=s["status"], boundary=c["boundary"])
    s["turn"] ^= 1
    return E, Ef


def run(s):
    c, kind = s["case"], s["kind"]
    if kind == "macro":
        ctx = s["ctx"]
        ctx.set_coarse(s["coarse"])
        ctx.step()
        return {"coarse": ctx.get_coarse(), "slope": ctx.get_slope()}
    if kind == "pic":
        s["ctx"].pic_steps(20)
        return {"measured": s["ctx"].measure()}
    if kind == "ensemble":
        s["batch"].step()
        return [x.view("coarse", torch.float64, 2 * x.cfg.n_coarse) for x in s["ctxs"]]
    if kind == "field":
        E, Ef = _solve(s)
        return {"E": E, "Ef": Ef, "phi": s["phi"]}
    if kind == "restrict":
        cell, theta, v, w = s["parts"]
        s_w, s_p = _restrict_shifts(c)
        pe.deposit(cell, theta, w, c["ncell"], s_w, rho=s["rho"], status=s["status"])
        args = pe.make_sample_args(s["E0f"], c["tau"], 1.0, 2.0, s_w, s_p, s["sample"], bin_shift=_bins(c))
        pe.sample(cell, theta, v, w, s["Ef"], c["ncell"], 0.1, 1.0, args, status=s["status"])
        coarse = pe.coarsen(s["sample"], 1, c["ncell"], s_w, s_p, c["n_coarse"], c["wavelet"], bin_shift=_bins(c))
        return {"rho": s["rho"], "sample": s["sample"], "coarse": coarse}
    if kind == "diag":
        return pe.compute_moments(*s["parts"], s["Ef"], c["ncell"], 0.5, 0.1, 0.1, 1.0, _shift(2.0 * c["ncell"] / c["N"]),
                                  phi=s["phi"], E=s["E"])
    if kind == "train":
        loss = s["net"].train(s["X"], s["Y"], c["B"], c["nsteps"], 1e-3, seed=s["seed"], shift_period=c["d"] // 2)
        return {"params": s["net"].params(), "loss": loss}
    with torch.cuda.stream(s["stream"]):
        return s["net"].forward(s["x"])  # the network's stream: training replays a graph on it


# ------------------------------------------------------------------ work


def work(case):
    c, kind = case, case["kind"]
    if kind == "macro":
        # particles do not fit on the chip: each fine step reads four and writes three values of
        # each, the lift writes four, the last sample reads four
        n = c["ncell"] * c["ppc"]
        species = 2 if c["electrons"] == "kinetic" else 1
        b = n * (28.0 * c["K"] * species + 16.0 * species + 16.0)
        return {"bytes": b, "flops": 60.0 * n * c["K"] * species}
    if kind == "pic":
        n = c["ncell"] * c["ppc"] * (2 if c["electrons"] == "kinetic" else 1)
        return {"bytes": n * (28.0 * 20 + 32.0 + 16.0), "flops": 40.0 * n * 20}
    if kind == "ensemble":
        n = sum(m[1] for m in _members(c))
        return {"bytes": n * (28.0 * c["K"] + 32.0), "flops": 60.0 * n * c["K"]}
    if kind == "field":
        return {"bytes": c["ncell"] * (8 + 8 + 8 + 8 + 4.0), "flops": 100.0 * c["ncell"]}
    if kind == "restrict":
        # one read of the particles serves the deposit and the sample
        return {"bytes": 16.0 * c["N"] + 32.0 * c["ncell"], "flops": 50.0 * c["N"]}
    if kind == "diag":
        return {"bytes": 16.0 * c["N"] + 20.0 * c["ncell"], "flops": 20.0 * c["N"]}
    dims = _dims(c)
    mm = sum(a * b for a, b in zip(dims[:-1], dims[1:]))
    if kind == "train":
        # forward, weight and data gradients; Adam reads and writes three FP32 values of each parameter
        per = 2.0 * c["B"] * (3 * mm - dims[0] * dims[1])
        return {"bytes": c["nsteps"] * (24.0 * mm + 8.0 * c["B"] * c["d"]), "flops": c["nsteps"] * per}
    return {"bytes": 2.0 * mm + c["B"] * c["d"] * (16.0 if c["f64"] else 8.0), "flops": 2.0 * c["B"] * mm}


# ------------------------------------------------------------------ 64-bit values


def exact(case, seed):
    kind = case["kind"]
    if kind == "field":
        return _exact_field(case, seed)
    if kind == "restrict":
        return _exact_restrict(case, seed)
    if kind == "diag":
        return _exact_diag(case, seed)
    if kind == "infer":
        return _exact_infer(case, seed)
    return None  # whole runs and trainings: every step's rounding travels through all that follow


def _thomas(a, b, c, d):
    """Tridiagonal solve a_j x_{j-1} + b_j x_j + c_j x_{j+1} = d_j (d: a list of right-hand sides)."""
    n = len(b)
    a, b, c = a.tolist(), b.tolist(), c.tolist()
    d = [x.tolist() for x in d]
    for j in range(1, n):
        m = a[j] / b[j - 1]
        b[j] -= m * c[j - 1]
        for x in d:
            x[j] -= m * x[j - 1]
    for x in d:
        x[n - 1] /= b[n - 1]
        for j in range(n - 2, -1, -1):
            x[j] = (x[j] - c[j] * x[j + 1]) / b[j]
    return [np.array(x) for x in d]


def _exact_field(c, seed):
    n, dx, walls = c["ncell"], c["dx"], c["boundary"] == "absorbing"
    rho = _density(c, _gen(seed))[0].cpu().numpy() * 2.0 ** -(FIELD_SHIFT + 24)
    if walls:
        rho[0] *= 2.0
        rho[-1] *= 2.0
    o = 1.0 / dx**2
    boltz = c["mode"] == "boltzmann"
    phi = np.log(np.maximum(rho, 1e-3)) if boltz else rho - 1.0

    def residual(p):
        left, right = np.roll(p, 1), np.roll(p, -1)
        if walls:
            left[0], right[-1] = p[1], p[-2]
        return (left - 2 * p + right) * o - (np.exp(p) if boltz else 1.0 + p) + rho

    for _ in range(60):
        lo, up = np.full(n, -o), np.full(n, -o)
        b = 2 * o + (np.exp(phi) if boltz else np.ones(n))
        r = residual(phi)
        if walls:
            up[0], lo[-1] = -2 * o, -2 * o
            step = _thomas(lo, b, up, [r])[0]
        else:  # cyclic corners by the Sherman-Morrison formula
            gam = -b[0]
            b[0] -= gam
            b[-1] -= o * o / gam
            u = np.zeros(n)
            u[0], u[-1] = gam, -o
            y, q = _thomas(lo, b, up, [r, u])
            f = -o / gam
            step = y - q * (y[0] + f * y[-1]) / (1.0 + q[0] + f * q[-1])
        m = np.max(np.abs(step))
        phi = phi + step * min(1.0, 2.0 / max(m, 1e-300))
        if m < 1e-13:
            break
    E = -(np.roll(phi, -1) - np.roll(phi, 1)) / (2 * dx)
    if walls:
        E[0] = E[-1] = 0.0
    return {"E": E, "Ef": E, "phi": phi}


def _exact_restrict(c, seed):
    (cell, theta, v, w), Ef, E0f = _restrict_inputs(c, seed)
    cell, theta, v, w, Ef, E0f = (t.cpu().numpy().astype(np.float64) if t.is_floating_point() else t.cpu().numpy()
                                  for t in (cell, theta, v, w, Ef, E0f))
    n = c["ncell"]
    nxt = (cell + 1) % n
    vbar = v + 0.5 * 0.1 * ((1 - theta) * Ef[cell] + theta * Ef[nxt])
    vt = vbar + c["tau"] * ((1 - theta) * E0f[cell] + theta * E0f[nxt])
    x = cell + theta + c["tau"] * 2.0 * vbar
    left = np.floor(x)
    f = x - left
    j0 = left.astype(np.int64) % n
    j1 = (j0 + 1) % n
    rows = []
    for q in (w, w * vt):
        a = (np.bincount(j0, q * (1 - f), n) + np.bincount(j1, q * f, n)) * 2.0 ** (-0.5 * math.log2(n))
        if c["wavelet"] == "d4":
            r3 = math.sqrt(3.0)
            h = np.array([1 + r3, 3 + r3, 3 - r3, 1 - r3]) / (4 * math.sqrt(2.0))
        else:
            h = np.array([1.0, 1.0]) / math.sqrt(2.0)
        while a.size > c["n_coarse"]:
            k = 2 * np.arange(a.size // 2)
            a = sum(h[m] * a[(k + m) % a.size] for m in range(h.size))
        rows.append(a)
    return {"rho": None, "sample": None, "coarse": np.stack(rows)[None]}


def _exact_diag(c, seed):
    s = prepare(c, seed)
    cell, theta, v, w = (t.cpu().numpy() for t in s["parts"])
    theta, v, w64 = theta.astype(np.float64), v.astype(np.float64), w.astype(np.float64)
    Ef, phi, E = (s[k].cpu().numpy().astype(np.float64) for k in ("Ef", "phi", "E"))
    n, dx = c["ncell"], 0.5
    vb = v + 0.5 * 0.1 * ((1 - theta) * Ef[cell] + theta * Ef[(cell + 1) % n])
    kin, fe = 0.5 * np.sum(w64 * vb * vb) * dx, 0.5 * np.sum(E * E) * dx
    ee = np.sum(phi * np.exp(phi) - np.exp(phi) + 1.0) * dx
    vmax = float(np.max(np.abs(vb)))
    return {"charge_fx": None, "invalid": None, "charge_wq": None,
            "charge_fixed_point": None,  # follows charge_fx, whose 64 bits wrap for many particles
            "charge": float(np.sum(w64) * dx),
            "momentum": None,  # a sum that nearly cancels: no scale of its own
            "kinetic": float(kin), "field_energy": float(fe), "electron_energy": float(ee),
            "total_energy": float(kin + fe + ee), "max_speed": vmax, "cfl": vmax * 0.1 / dx}


def _exact_infer(c, seed):
    g = _gen(seed)
    X, Y = _pairs(c, max(64, c["B"]), g)
    p = _weights(c, g).cpu().numpy().astype(np.float64)
    X, Y = X.cpu().numpy().astype(np.float64), Y.cpu().numpy().astype(np.float64)

    def stats(a):
        sd = a.std(axis=0)
        return a.mean(axis=0), np.maximum(sd, 1e-6 * sd.max())

    (mi, si), (mo, so) = stats(X), stats(Y)
    z, at, dims = torch.from_numpy((X[: c["B"]] - mi) / si), 0, _dims(c)
    for k, (a, b) in enumerate(zip(dims[:-1], dims[1:])):
        W = torch.from_numpy(p[at:at + a * b].reshape(b, a))
        z = z @ W.T + torch.from_numpy(p[at + a * b:at + a * b + b])
        at += a * b + b
        if k < len(dims) - 2:
            z = 0.5 * z * (1.0 + torch.erf(z / math.sqrt(2.0)))
    return z.numpy() * so + mo
