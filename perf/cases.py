"""The timed cases: what a user of this package has it compute, through its
public entry points (Plan, RealSpace, Batch, autograd.se_energy).

A case is a dict of plain values; `mode` says which entry point it goes
through:

  kspace    Plan.evaluate, results on the device
  host      Plan.energy_force_host_ptrs on page-locked host buffers
  ik        Plan.evaluate with forces by differentiation in Fourier space
  grad      autograd.se_energy, forward and backward
  real      RealSpace.evaluate, the erfc terms within rc and the self term
  ewald     the k-space sum, then the real-space sum added to its outputs
  ensemble  Batch.evaluate, many boxes in one call

Sizes are those of systems.WORKLOADS and of the benchmark's legs, and one
larger box of the same water; everything is evaluated with the package's
default settings.  Energies are FP64 scalars, forces and potentials have the
case's precision.
"""
import functools
import math
import random

import numpy as np
import torch

from paper_1712_04718_gb300 import autograd, se, systems

SHAPE_C = 0.95          # the plan's default shape constant (m = c sqrt(pi P))
XI = 3.12               # Ewald parameter of the water workloads, 1/nm
SPACING = 0.12          # their grid spacing, nm


def listed():
    water = dict(kind="water", xi=XI)
    return [
        # the 1000-charge test system at tight accuracy: the smallest call,
        # a few short kernels, launches and hand-overs
        dict(name="kspace-f64-1k", mode="kspace", kind="uniform", prec="fp64", N=1000, L=3.0,
             xi=3.5, M=32, P=16),
        # one MD step's k-space sum of an ordinary water box in single precision
        dict(name="kspace-f32-21k", mode="kspace", prec="fp32", L=6.0, M=52, P=8, **water),
        # the same step from and to page-locked host memory (an MD code on the CPU)
        dict(name="host-f32-21k", mode="host", prec="fp32", L=6.0, M=52, P=8, **water),
        # a large box on a grid the own transforms still take
        dict(name="kspace-f32-100k", mode="kspace", prec="fp32", L=10.0, M=84, P=8, **water),
        # a box beyond 128 grid points per dimension, on an odd grid
        dict(name="kspace-f32-410k", mode="kspace", prec="fp32", L=16.0, M=135, P=8, **water),
        # the ordinary box in double precision at the accuracy of single
        dict(name="kspace-f64-21k", mode="kspace", prec="fp64", L=6.0, M=52, P=8, **water),
        # the ordinary box as a reference calculation, to rounding
        dict(name="kspace-f64-21k-tight", mode="kspace", prec="fp64", L=6.0, M=96, P=24, **water),
        # forces that conserve momentum
        dict(name="ik-f32-21k", mode="ik", prec="fp32", L=6.0, M=52, P=8, **water),
        # training on the large box: energy, then the gradients by positions and charges
        dict(name="grad-f32-100k", mode="grad", prec="fp32", L=10.0, M=84, P=8, **water),
        # the real-space complement in double precision, 1 nm cut-off
        dict(name="real-f64-21k", mode="real", prec="fp64", L=6.0, rc=1.0, **water),
        # the whole Ewald sum of one MD step, parameters as select_params gives
        # them for an rms force error of 1e-3 of the rms force
        dict(name="ewald-f32-21k", mode="ewald", prec="fp32", kind="water", L=6.0, rc=0.94,
             xi=3.42, M=60, P=12),
        # many independent boxes of mixed sizes at once, at the support that
        # meets the workload's stated error
        dict(name="ensemble-f32-64", mode="ensemble", prec="fp32", kind="water", S=64, Lmin=3.0,
             Lmax=7.0, xi=XI, P=10),
    ]


def _eta(L, xi, M, P):
    return P * (L * xi / M) ** 2 / (SHAPE_C ** 2 * math.pi)


def _grid(rng, L, xi, P, lo=0.09, hi=0.13):
    """A grid for the box: any number of points (primes and odd ones among
    them) or the next 7-smooth one, fine enough for the support."""
    hi = min(hi, math.sqrt(0.62 * SHAPE_C ** 2 * math.pi / P) / xi)
    M = max(P, math.ceil(L / rng.uniform(min(lo, 0.75 * hi), hi)))
    return M if rng.random() < 0.5 else systems.smooth7(M)


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    top = max(work(c)["flops"] for c in listed())
    while True:
        case = _draw(rng)
        if work(case)["flops"] <= top:
            return case


def _draw(rng):
    mode = rng.choice(["kspace", "kspace", "kspace", "kspace", "host", "ik", "grad", "real",
                       "ewald", "ewald", "ensemble"])
    if mode == "ensemble":
        lo = rng.uniform(2.5, 5.0)
        return dict(mode=mode, prec="fp32", kind="water", S=int(_log(rng, 4, 65)),
                    Lmin=round(lo, 2), Lmax=round(rng.uniform(lo, 7.0), 2), xi=XI,
                    P=rng.choice([6, 8, 10]))
    prec = rng.choice(["fp32", "fp32", "fp64"])
    case = dict(mode=mode, prec=prec, kind=rng.choice(["water", "water", "uniform"]))
    big = {"kspace": 16.0, "host": 10.0, "ik": 7.0, "grad": 10.0, "real": 7.0, "ewald": 10.0}[mode]
    if prec == "fp64":
        big = min(big, 6.0)
    L = case["L"] = round(_log(rng, 2.2, big), 2)
    if case["kind"] == "uniform":
        case["N"] = int(100 * L ** 3 * rng.uniform(0.3, 1.0)) // 2 * 2
    if mode in ("real", "ewald"):
        case["rc"] = round(rng.uniform(0.6, min(1.1, L / 3.0 - 0.01)), 3)
        case["xi"] = round(rng.uniform(3.0, 3.4) / case["rc"], 3)
    else:
        case["xi"] = XI
    if mode != "real":
        case["P"] = rng.choice([4, 6, 8, 8, 10, 12, 16] if prec == "fp32"
                               else [6, 8, 10, 12, 16, 24])
        # the whole sum's xi is larger with a short cut-off, and its grid with it
        case["M"] = _grid(rng, L, case["xi"], case["P"], 0.28 / case["xi"], 0.41 / case["xi"])
    return case


def _boxes(case):
    """L and M of every box of an ensemble (the seed changes what is in them)."""
    r = np.random.Generator(np.random.PCG64(999))
    Ls = r.uniform(case["Lmin"], case["Lmax"], size=case["S"])
    return [(float(L), systems.smooth7(math.ceil(L / SPACING))) for L in Ls]


def _count(case, L=None):
    if case["kind"] == "uniform":
        return case["N"]
    return 3 * int(round(systems.WATER_DENSITY * (case["L"] if L is None else L) ** 3))


def _inputs(case, seed):
    dtype = np.float64 if case["prec"] == "fp64" else np.float32
    if case["kind"] == "uniform":
        return systems.uniform_charges(case["N"], case["L"], seed=seed, dtype=dtype)
    return systems.water_box(case["L"], seed=seed, dtype=dtype)


def _ensemble_inputs(case, seed):
    seed0 = random.Random(seed).randrange(1 << 40)
    return [systems.water_box(L, seed=seed0 + s, dtype=np.float32)
            for s, (L, _) in enumerate(_boxes(case))]


def prepare(case, seed):
    st = dict(case=case)
    if case["mode"] == "ensemble":
        boxes, parts = _boxes(case), _ensemble_inputs(case, seed)
        b = se.Batch([len(q) for _, q in parts], [L for L, _ in boxes], [M for _, M in boxes],
                     case["xi"], case["P"])
        st.update(batch=b, x=torch.tensor(np.concatenate([x for x, _ in parts]), device="cuda"),
                  q=torch.tensor(np.concatenate([q for _, q in parts]), device="cuda"),
                  F=torch.empty((b.Ntot, 3), device="cuda"), phi=torch.empty(b.Ntot, device="cuda"),
                  E=torch.empty(b.S, dtype=torch.float64, device="cuda"))
        return st
    x, q = _inputs(case, seed)
    N = len(q)
    if case["mode"] != "real":
        st["plan"] = se.Plan(N, case["L"], case["xi"], case["M"], case["P"], precision=case["prec"],
                             force_mode="ik" if case["mode"] == "ik" else "analytic")
    if case["mode"] in ("real", "ewald"):
        st["real"] = se.RealSpace(N, case["L"], case["xi"], case["rc"], precision=case["prec"])
    host = case["mode"] == "host"
    x, q = torch.from_numpy(x), torch.from_numpy(q)
    st["x"], st["q"] = (x.pin_memory(), q.pin_memory()) if host else (x.cuda(), q.cuda())
    if case["mode"] == "grad":
        st["x"].requires_grad_(True)
        st["q"].requires_grad_(True)
        return st
    where = dict(pin_memory=True) if host else dict(device="cuda")
    st["F"] = torch.empty((N, 3), dtype=x.dtype, **where)
    st["phi"] = torch.empty(N, dtype=x.dtype, **where)
    st["E"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    return st


def run(st):
    mode, x, q = st["case"]["mode"], st["x"], st["q"]
    if mode == "ensemble":
        E, F, phi = st["batch"].evaluate(x, q, st["F"], st["phi"], st["E"])
        return dict(E=E, F=F, phi=phi)
    if mode == "grad":
        E = autograd.se_energy(x, q, st["plan"])
        gx, gq = torch.autograd.grad(E, (x, q))
        return dict(E=E.detach(), gx=gx, gq=gq)
    F, phi, E = st["F"], st["phi"], st["E"]
    if mode == "host":
        E = st["plan"].energy_force_host_ptrs(x.data_ptr(), q.data_ptr(), F.data_ptr(),
                                              phi.data_ptr())
        return dict(E=E, F=F, phi=phi)
    if mode == "real":
        st["real"].evaluate(x, q, F, phi, E)
    else:
        st["plan"].evaluate(x, q, F, phi, E)
        if mode == "ewald":
            st["real"].evaluate(x, q, F, phi, E, accumulate=True)
    return dict(E=E, F=F, phi=phi)


def work(case):
    """Particles in, potentials and forces out; P^3 weights per particle
    spread (a multiply and an add each) and gathered (potential and force: two
    multiply-adds each, ik forces four), the transforms of the grid (one
    forward and one inverse, ik forces four inverse), and per pair within rc
    (taken once) 60 operations."""
    size = 8 if case["prec"] == "fp64" else 4
    ik = case["mode"] == "ik"

    def kspace(N, M, P):
        fft = 2.5 * M ** 3 * math.log2(M ** 3)
        return N * P ** 3 * (2 + (8 if ik else 4)) + (5 if ik else 2) * fft + 3.0 * M ** 3

    if case["mode"] == "ensemble":
        boxes = [(_count(case, L), M) for L, M in _boxes(case)]
        N = sum(n for n, _ in boxes)
        return dict(bytes=8 * size * N, flops=sum(kspace(n, M, case["P"]) for n, M in boxes))
    N = _count(case)
    flops = 0.0
    if case["mode"] != "real":
        flops += kspace(N, case["M"], case["P"])
    if case["mode"] in ("real", "ewald"):
        flops += 60 * 0.5 * N * N * (4 * math.pi / 3) * (case["rc"] / case["L"]) ** 3
    return dict(bytes=8 * size * N, flops=flops)


# ---- the same results in 64 bits, by plain torch ----

def _kspace64(x, q, L, xi, M, P, ik):
    """E, F, phi of the discrete Spectral Ewald sum for the given inputs; the
    cell of a particle is taken in the inputs' own precision, as the entry
    points document it, everything else in FP64."""
    eta = _eta(L, xi, M, P)
    alpha, h = 2 * xi * xi / eta, L / M
    cg = (2 * xi * xi / (math.pi * eta)) ** 1.5
    one = np.float64 if x.dtype == torch.float64 else np.float32
    cell = torch.floor(x * float(one(M / L))).clamp(0, M - 1).to(torch.int64)
    xd, qd = x.double(), q.double()
    a = torch.arange(P, device=x.device)
    N, step = len(q), max(1, (1 << 25) // P ** 3)

    def windows(s):
        pts = cell[s, :, None] - P // 2 + 1 + a                    # [n, 3, P]
        d = pts.double() * h - xd[s, :, None]
        g = torch.exp(-alpha * d * d)
        j = torch.remainder(pts, M)
        idx = ((j[:, 0, :, None, None] * M + j[:, 1, None, :, None]) * M + j[:, 2, None, None, :])
        return g, d * g, idx

    H = torch.zeros(M ** 3, dtype=torch.float64, device=x.device)
    for b in range(0, N, step):
        s = slice(b, min(N, b + step))
        g, _, idx = windows(s)
        w = (qd[s, None, None, None] * cg) * g[:, 0, :, None, None] * g[:, 1, None, :, None] \
            * g[:, 2, None, None, :]
        H.index_add_(0, idx.reshape(-1), w.reshape(-1))
    k = torch.fft.fftfreq(M, d=1.0 / M, device=x.device, dtype=torch.float64)
    kz = torch.arange(M // 2 + 1, device=x.device, dtype=torch.float64)
    k2 = (2 * math.pi / L) ** 2 * (k[:, None, None] ** 2 + k[None, :, None] ** 2
                                   + kz[None, None, :] ** 2)
    G = 4 * math.pi * torch.exp(-(1 - eta) * k2 / (4 * xi * xi)) / k2
    G[0, 0, 0] = 0.0
    S = torch.fft.rfftn(H.view(M, M, M)) * G
    grids = [torch.fft.irfftn(S, s=(M, M, M)).reshape(-1)]
    if ik:
        def nyq(v):   # the derivative's factor is 0 at the index whose sign is ambiguous
            return torch.where(2 * v.abs() == M, torch.zeros_like(v), v) * (2j * math.pi / L)
        for f in (nyq(k)[:, None, None], nyq(k)[None, :, None], nyq(kz)[None, None, :]):
            grids.append(torch.fft.irfftn(S * f, s=(M, M, M)).reshape(-1))
    phi = torch.empty(N, dtype=torch.float64, device=x.device)
    F = torch.empty(N, 3, dtype=torch.float64, device=x.device)
    h3 = h ** 3 * cg
    for b in range(0, N, step):
        s = slice(b, min(N, b + step))
        g, dg, idx = windows(s)

        def plain(grid):
            t = (grid[idx] * g[:, 2, None, None, :]).sum(-1)
            return ((t * g[:, 1, None, :]).sum(-1) * g[:, 0]).sum(-1)

        if ik:
            phi[s] = h3 * plain(grids[0])
            for c in range(3):
                F[s, c] = -h3 * qd[s] * plain(grids[1 + c])
            continue
        v = grids[0][idx]
        t, tz = (v * g[:, 2, None, None, :]).sum(-1), (v * dg[:, 2, None, None, :]).sum(-1)
        u, uy, uz = ((t * g[:, 1, None, :]).sum(-1), (t * dg[:, 1, None, :]).sum(-1),
                     (tz * g[:, 1, None, :]).sum(-1))
        phi[s] = h3 * (u * g[:, 0]).sum(-1)
        F[s] = (-2 * alpha * h3 * qd[s])[:, None] * torch.stack(
            [(u * dg[:, 0]).sum(-1), (uy * g[:, 0]).sum(-1), (uz * g[:, 0]).sum(-1)], 1)
    return 0.5 * (qd * phi).sum(), F, phi


def _real64(x, q, L, xi, rc):
    """E, F, phi of the erfc terms within rc and the self term."""
    xd, qd = x.double(), q.double()
    N, step = len(q), max(1, (1 << 26) // len(q))
    phi = -2 * xi / math.sqrt(math.pi) * qd
    F = torch.zeros(N, 3, dtype=torch.float64, device=x.device)
    for b in range(0, N, step):
        r2 = 0.0
        for c in range(3):
            d = xd[b:b + step, None, c] - xd[None, :, c]
            r2 = r2 + (d - L * torch.round(d / L)) ** 2
        i, j = torch.nonzero((r2 < rc * rc) & (r2 > 0), as_tuple=True)
        d = xd[b + i] - xd[j]
        d = d - L * torch.round(d / L)
        r2 = (d * d).sum(1)
        r = r2.sqrt()
        e = torch.special.erfc(xi * r) / r
        phi.index_add_(0, b + i, qd[j] * e)
        f = qd[b + i] * qd[j] * (2 * xi / math.sqrt(math.pi) * torch.exp(-xi * xi * r2) + e) / r2
        F.index_add_(0, b + i, f[:, None] * d)
    return 0.5 * (qd * phi).sum(), F, phi


def exact(case, seed):
    if case["mode"] == "ensemble":
        parts = [_kspace64(torch.tensor(x, device="cuda"), torch.tensor(q, device="cuda"), L,
                           case["xi"], M, case["P"], False)
                 for (x, q), (L, M) in zip(_ensemble_inputs(case, seed), _boxes(case))]
        return dict(E=torch.stack([p[0] for p in parts]), F=torch.cat([p[1] for p in parts]),
                    phi=torch.cat([p[2] for p in parts]))
    x, q = (torch.from_numpy(v).cuda() for v in _inputs(case, seed))
    sums = []
    if case["mode"] != "real":
        sums.append(_kspace64(x, q, case["L"], case["xi"], case["M"], case["P"],
                              case["mode"] == "ik"))
    if case["mode"] in ("real", "ewald"):
        sums.append(_real64(x, q, case["L"], case["xi"], case["rc"]))
    E, F, phi = (functools.reduce(torch.add, v) for v in zip(*sums))
    if case["mode"] == "grad":
        return dict(E=E, gx=-F, gq=phi)
    if case["mode"] == "host":
        return dict(E=float(E), F=F.cpu(), phi=phi.cpu())
    return dict(E=E.reshape(1), F=F, phi=phi)
