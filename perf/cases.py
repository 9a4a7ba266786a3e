"""Timed cases of the library: what its users have it do, through its Python entry points.

A case is one operation on one state point (or a batch of them):

  map        G(rho) of a caller that drives its own fixed-point scheme (``Plan.picard_map``)
  fields     the weighted densities, both one-body correlations and psi of a given density
  iterate    K Picard iterations queued on the device (``iter_begin`` + ``iter_run``)
  solve      Picard iterations to a tolerance, the residual read every iteration
  newton     the Newton-Krylov solver to a tolerance
  step_host  one Picard step on host buffers (copies in and out included)
  grad       the grand potential and its three gradients through autograd
  batch      K iterations of a ragged batch of state points

The geometries are hard neutral spheres, a planar wall, a charged pore through a slab or a smooth
field, on grids whose lengths have compile-time kernels and on others, in FP32 and FP64.  Inputs
are made on the GPU from the seed.  ``exact`` restates the method in FP64 with torch alone.
"""
import math

import numpy as np
import torch

from paper_0910_1531_gb300 import autograd, binding

PER_NM3 = 0.602214076                      # mol/L -> nm^-3
SPECIES = {                                # radius (nm), valence
    "Na": (0.095, 1.0), "Cl": (0.181, -1.0), "Ca": (0.099, 2.0), "O": (0.14, -0.5),
    "cation": (0.1, 1.0), "anion": (0.2125, -1.0), "HS": (0.1, 0.0),
}


def listed():
    return [
        # the smallest call: one G of a 32^3 salt around a sphere, where launches are all that counts
        {"name": "map_32", "op": "map", "geometry": "spheres", "nx": 32, "ny": 32, "nz": 32, "h": 0.1,
         "species": "Na Cl", "molar": "0.1 0.1", "obstacles": 1, "precision": "fp32"},
        # the plain FP64 small configuration: 50 fixed-mixing iterations at 32^3
        {"name": "iterate_32_f64", "op": "iterate", "geometry": "spheres", "nx": 32, "ny": 32, "nz": 32, "h": 0.1,
         "species": "Na Cl", "molar": "0.1 0.1", "obstacles": 1, "precision": "fp64", "iters": 50, "alpha": 0.1},
        # post-processing of a density on a ragged box without compile-time lengths, odd in y
        {"name": "fields_120x75x84", "op": "fields", "geometry": "spheres", "nx": 120, "ny": 75, "nz": 84, "h": 0.06,
         "species": "Na Cl", "molar": "0.5 0.5", "obstacles": 6, "precision": "fp32"},
        # the differentiated form: 0.5 M salt in a smooth field, forward and backward
        {"name": "grad_64", "op": "grad", "geometry": "smooth", "nx": 64, "ny": 64, "nz": 64, "h": 0.1,
         "species": "Na Cl", "molar": "0.5 0.5", "precision": "fp32"},
        # the paper's ionic calculation at a hard wall, to convergence in FP64 (odd lengths 21 and 161)
        {"name": "wall_21x21x161_f64", "op": "solve", "geometry": "wall", "nx": 21, "ny": 21, "nz": 161, "h": 0.09523809523809523,
         "hz": 0.037267080745341616, "species": "cation anion", "molar": "1.0 1.0", "precision": "fp64", "alpha": -1.0,
         "tol": 1e-8, "iters": 2000},
        # dense hard spheres at a hard wall, one species, Newton-Krylov in FP64 on a thin box
        {"name": "newton_4x4x512_f64", "op": "newton", "geometry": "wall", "nx": 4, "ny": 4, "nz": 512, "h": 0.05, "hz": 0.00625,
         "species": "HS", "packing": 0.4, "precision": "fp64", "tol": 1e-10, "iters": 50},
        # the headline: three species around sixteen obstacles, line search, on an autotuned plan
        {"name": "iterate_128", "op": "iterate", "geometry": "spheres", "nx": 128, "ny": 128, "nz": 128, "h": 0.05,
         "species": "Na Ca Cl", "molar": "0.1 0.01 0.12", "obstacles": 16, "precision": "fp32", "iters": 10, "alpha": -1.0,
         "autotune": True},
        # the same in plain FP64
        {"name": "iterate_128_f64", "op": "iterate", "geometry": "spheres", "nx": 128, "ny": 128, "nz": 128, "h": 0.05,
         "species": "Na Ca Cl", "molar": "0.1 0.01 0.12", "obstacles": 16, "precision": "fp64", "iters": 3, "alpha": -1.0},
        # the step of a host program that keeps its fields in host memory
        {"name": "step_host_128", "op": "step_host", "geometry": "spheres", "nx": 128, "ny": 128, "nz": 128, "h": 0.05,
         "species": "Na Ca Cl", "molar": "0.1 0.01 0.12", "obstacles": 16, "precision": "fp32", "alpha": -1.0},
        # a resolution chosen by its spacing and not by its radix: 160^3, line search
        {"name": "iterate_160", "op": "iterate", "geometry": "spheres", "nx": 160, "ny": 160, "nz": 160, "h": 0.04,
         "species": "Na Ca Cl", "molar": "0.1 0.01 0.12", "obstacles": 16, "precision": "fp32", "iters": 5, "alpha": -1.0},
        # the large configuration: four species, one of them a fixed number of ions in a pore, on an
        # autotuned plan
        {"name": "pore_256", "op": "iterate", "geometry": "pore", "nx": 256, "ny": 256, "nz": 256, "h": 0.05,
         "species": "Na Ca Cl O", "molar": "0.1 0.001 0.102 0", "fixed": 8.0, "precision": "fp32", "iters": 5,
         "alpha": 0.05, "autotune": True},
        # many state points at once, ragged sizes, on autotuned plans
        {"name": "batch_16", "op": "batch", "sizes": "32 48 64 96 64 32 96 48 48 64 32 96 64 48 32 64", "h": 0.1,
         "precision": "fp32", "iters": 10, "alpha": -1.0, "autotune": True},
    ]


# ---------------------------------------------------------------------------------- draws
def _valid(n):
    for p in (2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31):
        while n % p == 0:
            n //= p
    return n == 1


_LENGTHS = [n for n in range(20, 225) if _valid(n)]
_NICE = [n for n in _LENGTHS if n % 4 == 0 and max(p for p in (2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31) if n % p == 0) <= 7]


def _length(rng, lo, hi, pool):
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(pool, key=lambda n: abs(math.log(n / x)))


def draw(rng):
    """One more case: op, sizes (their logarithm uniform; half of the boxes cubic, some lengths
    odd), species, precision and form of the hard-sphere functional."""
    op = rng.choice(["map", "fields", "iterate", "iterate", "grad", "solve", "step_host", "batch"])
    f64 = rng.random() < 0.3
    c = {"op": op, "precision": "fp64" if f64 else "fp32"}
    if op == "batch":
        count = rng.randint(3, 20)
        top = 64 if f64 else 110
        c.update(sizes=" ".join(str(_length(rng, 20, top, _LENGTHS)) for _ in range(count)),
                 h=round(rng.uniform(0.06, 0.1), 4), iters=rng.randint(2, 10), alpha=-1.0)
        return c
    top = 128 if f64 else 224
    if rng.random() < 0.5:
        n = _length(rng, 24, top, _NICE if rng.random() < 0.7 else _LENGTHS)
        c.update(nx=n, ny=n, nz=n)
    else:
        c.update({k: _length(rng, 20, top, _LENGTHS) for k in ("nx", "ny", "nz")})
    salt = round(math.exp(rng.uniform(math.log(0.02), math.log(0.5))), 4)
    species, molar = rng.choice([
        ("HS", f"{round(20.0 * salt, 4)}"), ("Na Cl", f"{salt} {salt}"), ("Na Cl", f"{salt} {salt}"),
        ("Na Ca Cl", f"{salt} {round(salt / 8, 4)} {round(salt + 2 * round(salt / 8, 4), 4)}"),
        ("Na Ca Cl cation", f"{salt} {round(salt / 8, 4)} {round(2 * salt + 2 * round(salt / 8, 4), 4)} {salt}")])
    c.update(geometry="smooth" if op == "grad" or rng.random() < 0.2 else "spheres", h=round(rng.uniform(0.04, 0.1), 4),
             species=species, molar=molar, obstacles=rng.randint(1, 8),
             functional=rng.choice(["rslt", "rslt", "rslt", "white_bear", "rosenfeld"]))
    if op in ("iterate", "solve"):
        c.update(iters=rng.randint(2, 6), alpha=rng.choice([-1.0, -1.0, 0.1]))
        if op == "solve":
            c["tol"] = 0.0
    elif op == "step_host":
        c["alpha"] = -1.0
    return c


# ---------------------------------------------------------------------------------- inputs
def _shape(c):
    return (c["nz"], c["ny"], c["nx"])


def _spacing(c):
    return (c["h"], c["h"], c.get("hz", c["h"]))


def _species_of(c):
    names = c["species"].split()
    radius = [SPECIES[n][0] for n in names]
    valence = [SPECIES[n][1] for n in names]
    if "packing" in c:
        molar = [c["packing"] / (4.0 / 3.0 * math.pi * radius[0] ** 3) / PER_NM3]
    else:
        molar = [float(m) for m in c["molar"].split()]
    return radius, valence, molar


def _generator(seed, dev):
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) * 7919 + 13)
    return g


def _smooth(shape, h, length, gen, dev):
    """Zero-mean Gaussian random field of unit variance, correlation length `length` (nm)."""
    white = torch.randn(shape, generator=gen, device=dev, dtype=torch.float64)
    k = _kgrid(shape, h, dev)
    f = torch.fft.irfftn(torch.fft.rfftn(white) * torch.exp(-0.25 * k["k2"] * length ** 2), s=shape)
    f = f - f.mean()
    return f / f.std()


def _axes(shape, h, dev):
    (nz, ny, nx), (hx, hy, hz) = shape, h
    a = lambda n, d: torch.arange(n, device=dev, dtype=torch.float64) * d
    return a(nz, hz)[:, None, None], a(ny, hy)[None, :, None], a(nx, hx)[None, None, :]


def _near(d, length):
    return d - length * torch.round(d / length)


def _potential(c, gen, dev):
    """V (S, nz, ny, nx) in FP64: +inf where a species is excluded."""
    shape, h = _shape(c), _spacing(c)
    radius, valence, _ = _species_of(c)
    S = len(radius)
    z, y, x = _axes(shape, h, dev)
    L = (shape[2] * h[0], shape[1] * h[1], shape[0] * h[2])
    V = torch.zeros((S,) + shape, device=dev, dtype=torch.float64)
    kind = c["geometry"]
    if kind == "smooth":
        f = _smooth(shape, h, 0.5, gen, dev)
        for i in range(S):
            V[i] = (valence[i] if valence[i] else 0.7) * f
    elif kind == "spheres":
        # non-overlapping hard neutral spheres that together leave most of the box free
        n = c["obstacles"]
        top = 0.45 * (min(L) if n == 1 else min(min(L), (L[0] * L[1] * L[2] / n) ** (1.0 / 3.0)))
        u = torch.rand((400, 4), generator=gen, device=dev, dtype=torch.float64).cpu().numpy()
        done = []
        for r in u:
            R = top * (0.4 + 0.4 * r[3])
            p = [float(L[d] * r[d]) for d in range(3)]
            if all(math.sqrt(sum((a - b - l * round((a - b) / l)) ** 2 for a, b, l in zip(p, q, L))) >= R + Q for q, Q in done):
                done.append((p, R))
                if len(done) == n:
                    break
        for p, R in done:
            r2 = _near(x - p[0], L[0]) ** 2 + _near(y - p[1], L[1]) ** 2 + _near(z - p[2], L[2]) ** 2
            for i in range(S):
                V[i].masked_fill_(r2 < (R + radius[i]) ** 2, math.inf)
    elif kind == "wall":
        d = _near(z, L[2]).abs().expand(shape)
        for i in range(S):
            V[i].masked_fill_(d < radius[i], math.inf)
    else:   # pore: a 2 nm slab with a cylindrical hole; the last species confined to its middle
        rp = torch.sqrt(_near(x - L[0] / 2, L[0]) ** 2 + _near(y - L[1] / 2, L[1]) ** 2)
        dz = _near(z - L[2] / 2, L[2]).abs()
        for i in range(S - 1):
            V[i].masked_fill_(((dz < 1.0 + radius[i]) & (rp > 0.5 - radius[i])).expand(shape), math.inf)
        V[S - 1].masked_fill_(~((rp <= 0.5 - radius[-1]) & (dz <= 0.5 - radius[-1])).expand(shape), math.inf)
    return V


def _fixed(c):
    return [0.0] * (len(c["species"].split()) - 1) + [c["fixed"]] if "fixed" in c else None


def _density(c, V, gen, dev):
    """A positive density in FP64: the bath (a fixed-number species its particles spread over its
    voxels) times a seeded smooth modulation, zero on excluded voxels."""
    shape, h = _shape(c), _spacing(c)
    _, _, molar = _species_of(c)
    fixed = _fixed(c)
    # given densities vary like a profile; the start of an iteration is near the bath
    amp = 0.3 if c["op"] in ("map", "fields", "grad") else 0.05
    rho = torch.empty_like(V)
    for i, m in enumerate(molar):
        f = 1.0 + amp * torch.tanh(_smooth(shape, h, 4.0 * max(h), gen, dev))
        free = ~torch.isinf(V[i])
        rho[i] = torch.where(free, f, torch.zeros_like(f))
        if fixed and fixed[i] > 0:
            rho[i] *= fixed[i] / (rho[i].sum() * h[0] * h[1] * h[2])
        else:
            rho[i] *= m * PER_NM3
    return rho


def _inputs(c, seed):
    dev = torch.device("cuda")
    gen = _generator(seed, dev)
    V = _potential(c, gen, dev)
    return _density(c, V, gen, dev), V


def _members(c, seed):
    """The state points of a batch, as cases of their own."""
    out = []
    rng = np.random.default_rng(int(seed) + 5)
    for n in (int(v) for v in c["sizes"].split()):
        m = round(float(np.exp(rng.uniform(math.log(0.01), math.log(0.3)))), 5)
        out.append({"op": "iterate", "geometry": "spheres", "nx": n, "ny": n, "nz": n, "h": c["h"], "species": "Na Cl",
                    "molar": f"{m} {m}", "obstacles": 1, "precision": c["precision"], "iters": c["iters"], "alpha": c["alpha"]})
    return out


def prepare(case, seed):
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    if case["op"] == "batch":
        members = _members(case, seed)
        fields = [_inputs(m, seed * 101 + i) for i, m in enumerate(members)]
        states = []
        for m in members:
            radius, valence, molar = _species_of(m)
            states.append({"shape": _shape(m), "h": _spacing(m), "radius": radius, "valence": valence, "bulk_molar": molar})
        s = {"case": case, "rho0": [r.to(dtype) for r, _ in fields], "V": [v.to(dtype) for _, v in fields],
             "batch": binding.Batch(states, precision=case["precision"])}
        s["rho"] = [r.clone() for r in s["rho0"]]
        if case.get("autotune"):
            s["batch"].autotune(s["rho"], s["V"])
        return s
    rho, V = _inputs(case, seed)
    rho, V = rho.to(dtype), V.to(dtype)
    radius, valence, molar = _species_of(case)
    plan = binding.Plan(_shape(case), _spacing(case), radius, valence, molar, precision=case["precision"],
                        n_fixed=_fixed(case), functional=case.get("functional", "rslt"))
    s = {"case": case, "plan": plan, "rho0": rho, "V": V}
    if case["op"] == "step_host":
        s["rho_host0"] = rho.cpu().pin_memory()
        s["V_host"] = V.cpu().pin_memory()
        s["rho_host"] = s["rho_host0"].clone().pin_memory()
    elif case["op"] == "grad":
        s["rho"] = rho.clone().requires_grad_(True)
        s["V"] = V.clone().requires_grad_(True)
        s["bath"] = torch.tensor(plan.bulk()["rho"], dtype=torch.float64, requires_grad=True)
    else:
        s["rho"] = rho.clone()
    if case.get("autotune"):
        plan.autotune(s["rho"], s["V"])
    return s


def run(state):
    c = state["case"]
    op = c["op"]
    if op == "batch":
        for r, r0 in zip(state["rho"], state["rho0"]):
            r.copy_(r0)
        state["batch"].begin(state["rho"], state["V"])
        state["batch"].iterate(c["iters"], c["alpha"])
        return {"rho": list(state["rho"])}
    plan = state["plan"]
    if op == "map":
        return {"G": plan.picard_map(state["rho"], state["V"], resid=False)}
    if op == "fields":
        c_es, psi = plan.c1_es(state["rho"], want_psi=True)
        return {"n": plan.weighted_densities(state["rho"]), "c1_hs": plan.c1_hs(state["rho"]), "c1_es": c_es, "psi": psi}
    if op == "grad":
        omega = autograd.grand_potential(plan, state["rho"], state["V"], state["bath"])
        d_rho, d_V, d_bath = torch.autograd.grad(omega, (state["rho"], state["V"], state["bath"]))
        return {"omega": omega.detach(), "d_rho": d_rho, "d_V": d_V, "d_bath": d_bath}
    if op == "step_host":
        # the host program's next density: it overwrites its own buffer
        state["rho_host"].copy_(state["rho_host0"])
        r, a = plan.picard_step_host(state["rho_host"], state["V_host"], c["alpha"])
        return {"rho": state["rho_host"], "resid": r, "alpha": a}
    rho = state["rho"]
    rho.copy_(state["rho0"])
    if op == "iterate":
        plan.iter_begin(rho, state["V"])
        # the residual is read, as a program does to decide whether to go on; near convergence it is
        # rounding noise, so the iterate is what is compared
        plan.iter_run(rho, state["V"], c["iters"], c["alpha"])
        return {"rho": rho}
    if op == "solve":
        plan.solve(rho, state["V"], c["tol"], c["iters"], c["alpha"])
        return {"rho": rho}
    plan.solve_newton(rho, state["V"], c["tol"], c["iters"])
    return {"rho": rho}


# ---------------------------------------------------------------------------------- what a pass needs
def work(case):
    """Bytes: the fields the caller hands over and gets back, once per pass (an iteration reads its
    iterate and V and writes the new iterate).  Flops: 2.5 N log2 N for each real 3D transform, S + 10
    for the weighted densities (ten of them inverse) and 10 + S for the correlations of every G."""
    if case["op"] == "batch":
        parts = [work(m) for m in _members(case, 0)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    N = case["nx"] * case["ny"] * case["nz"]
    S = len(case["species"].split())
    b = 8 if case["precision"] == "fp64" else 4
    half = 2.5 * N * math.log2(N) * (S + 10)          # one direction of one G
    op = case["op"]
    if op == "map":
        return {"bytes": 3 * S * N * b, "flops": 2 * half}
    if op == "fields":
        return {"bytes": (3 * S + 11) * N * b, "flops": 2 * half + 2.5 * N * math.log2(N) * (2 * S + 1)}
    if op == "grad":
        return {"bytes": 4 * S * N * b, "flops": 2 * half}
    # the converging solvers: the iterations (or evaluations) they need are not known here; ten
    k = 1 if op == "step_host" else (10 if case.get("tol") else case["iters"])
    per = 2 * half if (op == "newton" or case["alpha"] >= 0) else 4 * half
    return {"bytes": (k + 1) * 3 * S * N * b, "flops": 2 * half + k * per}


def tolerance(case):
    """The rounding of the transforms (about 30 passes) and of the exponent.  Against `exact`, FP32
    is off by 5e-8 (an iterate) to 4e-7 (the correlations of small-amplitude densities), FP64 by
    2e-16 to 1e-13.  A converged solve is compared at its stopping tolerance."""
    if case["op"] in ("solve", "newton") and case.get("tol"):
        return {"rel": 30 * case["tol"], "max": 3000 * case["tol"]}
    if case["precision"] == "fp64":
        return {"rel": 1e-12, "max": 1e-10}
    return {"rel": 4e-6, "max": 2e-4}


# ---------------------------------------------------------------------------------- the method in 64 bits
def _kgrid(shape, h, dev):
    """Wave numbers of the half spectrum (x halved), |k|^2 and the Nyquist masks of the three axes."""
    nz, ny, nx = shape

    def axis(n, d, half):
        j = torch.arange(n // 2 + 1 if half else n, device=dev, dtype=torch.float64)
        k = torch.where(2 * j <= n, j, j - n) * (2 * math.pi / (n * d))
        return k, (2 * j == n)

    (kz, qz), (ky, qy), (kx, qx) = axis(nz, h[2], False), axis(ny, h[1], False), axis(nx, h[0], True)
    kz, ky, kx = kz[:, None, None], ky[None, :, None], kx[None, None, :]
    lap = sum(4 * torch.sin(0.5 * k * d) ** 2 / d ** 2 for k, d in ((kx, h[0]), (ky, h[1]), (kz, h[2])))
    # the odd kernels have no component along an axis at that axis's Nyquist index
    return {"kx": kx * ~qx[None, None, :], "ky": ky * ~qy[None, :, None], "kz": kz * ~qz[:, None, None],
            "k2": kx * kx + ky * ky + kz * kz, "lap": lap}


def _ball(y, n):
    """sum_m (-1)^m y^(2m) / ((2m + 1)! (2m + n + 3)), summed for small y."""
    out, f = torch.zeros_like(y), 1.0
    for m in range(14):
        if m:
            f *= 2 * m * (2 * m + 1)
        out += (-1) ** m * y ** (2 * m) / (f * (2 * m + n + 3))
    return out


def _msa(rho, sigma, z, lb):
    """The MSA screening parameter (bisection) and the electrostatic bath potentials."""
    delta = 1 - math.pi / 6 * float(np.sum(rho * sigma ** 3))

    def eta(g):
        om = 1 + math.pi / (2 * delta) * float(np.sum(rho * sigma ** 3 / (1 + g * sigma)))
        return math.pi / (2 * delta * om) * float(np.sum(rho * sigma * z / (1 + g * sigma)))

    hi = math.sqrt(4 * math.pi * lb * float(np.sum(rho * z * z)))
    if hi == 0:
        return 0.0, np.zeros_like(rho)
    f = lambda g: g * g - math.pi * lb * float(np.sum(rho * ((z - eta(g) * sigma ** 2) / (1 + g * sigma)) ** 2))
    lo = 0.0
    while f(hi) <= 0:
        hi *= 2
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if f(mid) < 0 else (lo, mid)
    g = 0.5 * (lo + hi)
    e = eta(g)
    return g, -lb * (g * z * z / (1 + g * sigma) + e * sigma * ((2 * z - e * sigma ** 2) / (1 + g * sigma) + e * sigma ** 2 / 3))


def _phi(n, kind, want):
    """Phi (want "value") or its ten derivatives of the hard-sphere form `kind` at fields n (10, ...)."""
    n0, n1, n2, n3 = n[0], n[1], n[2], n[3]
    v1, v2 = n[4:7], n[7:10]
    D = 1 - n3
    q, dot = (v2 * v2).sum(0), (v1 * v2).sum(0)
    if kind == "rslt":
        ok = n2 > 1e-30
        xi = torch.where(ok, q / torch.where(ok, n2 * n2, torch.ones_like(n2)), torch.ones_like(n2)).clamp(0, 1)
        om = 1 - xi
        if want == "value":
            return -n0 * torch.log(D) + (n1 * n2 - dot) / D + (n2 * om) ** 3 / (24 * math.pi * D * D)
        d2 = n2 * n2 * om * om * (1 + xi) / (8 * math.pi * D * D)
        d3 = (n2 * om) ** 3 / (12 * math.pi * D ** 3)
        cv = n2 * om * om / (4 * math.pi * D * D)
    else:
        if kind == "rosenfeld":
            g, dg, w = torch.ones_like(D), torch.zeros_like(D), 24 * math.pi
        else:   # white_bear: g = (n3 + D^2 ln D) / n3^2, by its power series for small n3
            small = n3 < 0.4
            t, u = torch.where(small, n3, torch.zeros_like(n3)), torch.where(small, torch.full_like(n3, 0.5), n3)
            gs, ds = torch.full_like(t, 1.5), torch.zeros_like(t)
            p = torch.ones_like(t)
            for k in range(3, 50):
                gs = gs - 2 * p * t / (k * (k - 1) * (k - 2))
                ds = ds - 2 * p / (k * (k - 1))
                p = p * t
            e = 1 - u
            num = u + e * e * torch.log(e)
            g = torch.where(small, gs, num / u ** 2)
            dg = torch.where(small, ds, (u - 2 * e * torch.log(e)) / u ** 2 - 2 * num / u ** 3)
            w = 36 * math.pi
        f, df = g / (w * D * D), (dg * D + 2 * g) / (w * D ** 3)
        T = n2 ** 3 - 3 * n2 * q
        if want == "value":
            return -n0 * torch.log(D) + (n1 * n2 - dot) / D + T * f
        d2, d3, cv = 3 * (n2 * n2 - q) * f, T * df, 6 * n2 * f
    return torch.cat([torch.stack([-torch.log(D), n2 / D, n1 / D + d2, n0 / D + (n1 * n2 - dot) / (D * D) + d3]),
                      -v2 / D, -v1 / D - cv * v2])


class _Exact:
    """One state point's method in FP64, with torch's transforms."""

    def __init__(self, c, molar=None):
        self.c, self.shape, self.h = c, _shape(c), _spacing(c)
        dev = torch.device("cuda")
        radius, valence, m = _species_of(c)
        self.R, self.z = np.array(radius), np.array(valence)
        self.molar = np.array(m if molar is None else molar)
        self.S, self.kind = len(radius), c.get("functional", "rslt")
        rho, sigma = self.molar * PER_NM3, 2 * self.R
        self.rho_b = rho
        # the Bjerrum length at 298.15 K and eps_r = 78.5
        self.lb = 1.602176634e-19 ** 2 / (4 * math.pi * 8.8541878128e-12 * 78.5 * 1.380649e-23 * 298.15) * 1e9
        w = np.stack([np.ones(self.S), self.R, 4 * math.pi * self.R ** 2, 4 * math.pi * self.R ** 3 / 3])
        uniform = torch.tensor(np.concatenate([w @ rho, np.zeros(6)]), dtype=torch.float64)
        # mu_HS of the bath: the uniform limit of the functional (Percus-Yevick for the first two)
        self.mu_hs = _phi(uniform, self.kind, "derivatives")[:4].numpy() @ w
        self.gamma, self.mu_es = _msa(rho, sigma, self.z, self.lb)
        self.fixed = np.array(_fixed(c) or [0.0] * self.S)
        self.N = self.shape[0] * self.shape[1] * self.shape[2]
        self.dv = self.h[0] * self.h[1] * self.h[2]
        self.ref = np.where(self.fixed > 0, self.fixed / (self.N * self.dv), rho)
        self.k = _kgrid(self.shape, self.h, dev)
        k = torch.sqrt(self.k["k2"])
        self.w0, self.j3, self.K = [], [], {}
        for R in self.R:
            x = k * R
            small = x < 0.5
            xs = torch.where(small, torch.ones_like(x), x)
            self.w0.append(torch.sinc(x / math.pi))
            self.j3.append(torch.where(small, _ball(x * small, 0), (torch.sin(xs) - xs * torch.cos(xs)) / xs ** 3))
        zero = self.k["lap"] == 0
        inv_lap = torch.where(zero, torch.zeros_like(self.k["lap"]), 1 / torch.where(zero, torch.ones_like(self.k["lap"]), self.k["lap"]))
        self.psi_k = 4 * math.pi * self.lb * inv_lap
        for i in range(self.S):
            for j in range(i, self.S):
                R = self.R[i] + self.R[j]
                y = k * R
                small = y < 0.5
                ys = torch.where(small, torch.ones_like(y), y)
                s, co = torch.sin(ys), torch.cos(ys)
                om = 2 * torch.sin(0.5 * ys) ** 2
                b = [torch.where(small, _ball(y * small, n), v) for n, v in
                     ((-1, om / ys ** 2), (0, (s - ys * co) / ys ** 3), (1, -co / ys ** 2 + 2 * s / ys ** 3 - 2 * om / ys ** 4))]
                li, lj = (self.R[q] + 0.5 / self.gamma if self.gamma > 0 else math.inf for q in (i, j))
                a1, a0, am = (0.5 / (li * lj), 1 / li + 1 / lj, (li - lj) ** 2 / (2 * li * lj) + 2) if self.gamma > 0 else (0, 0, 2)
                self.K[i, j] = self.K[j, i] = 2 * math.pi * self.lb * self.z[i] * self.z[j] * R * R * (
                    a1 * R * R * b[2] - a0 * R * b[1] + am * b[0])

    def fwd(self, f):
        return torch.fft.rfftn(f, dim=(-3, -2, -1))

    def inv(self, f):
        return torch.fft.irfftn(f, s=self.shape, dim=(-3, -2, -1))

    def weighted(self, rho):
        acc = [0.0] * 5
        for i, R in enumerate(self.R):
            r = self.fwd(rho[i])
            for a, w in enumerate((self.w0[i], R * self.w0[i], 4 * math.pi * R * R * self.w0[i],
                                   4 * math.pi * R ** 3 * self.j3[i], R * R * self.j3[i])):
                acc[a] = acc[a] + r * w
        out = [self.inv(a) for a in acc[:4]]
        for a in (acc[4], acc[3]):                      # n_V1 = grad m, n_V2 = grad n3
            out += [self.inv(1j * self.k[d] * a) for d in ("kx", "ky", "kz")]
        return torch.stack(out)

    def c1_hs(self, n):
        d = _phi(n, self.kind, "derivatives")
        f = [self.fwd(d[a]) for a in range(4)]
        div = [sum(-1j * self.k[q] * self.fwd(d[o + a]) for a, q in enumerate(("kx", "ky", "kz"))) for o in (4, 7)]
        return torch.stack([-self.inv(self.w0[i] * (f[0] + R * f[1] + 4 * math.pi * R * R * f[2]) +
                                      self.j3[i] * (4 * math.pi * R ** 3 * (f[3] + div[1]) + R * R * div[0]))
                            for i, R in enumerate(self.R)])

    def screening(self, rho):
        """E_i = sum_j DC_ij (*) drho_j, and psi."""
        f = [self.fwd(r) for r in rho]
        psi = self.inv(sum(z * r for z, r in zip(self.z, f)) * self.psi_k)
        for j in range(self.S):
            f[j][0, 0, 0] -= self.N * self.rho_b[j]
        return torch.stack([self.inv(sum(self.K[i, j] * f[j] for j in range(self.S))) for i in range(self.S)]), psi

    def _col(self, v):
        return torch.as_tensor(v, dtype=torch.float64, device="cuda")[:, None, None, None]

    def G(self, rho, V):
        E, psi = self.screening(rho)
        c = self.c1_hs(self.weighted(rho)) + E - self._col(self.z) * psi
        g = self._col(self.rho_b) * torch.exp(self._col(self.mu_hs) - V + c)
        for i in np.flatnonzero(self.fixed > 0):
            e = torch.exp(-V[i] + c[i])
            g[i] = self.fixed[i] * e / (self.dv * e.sum())
        return g

    def resid2(self, rho, g):
        return float((((rho - g) / self._col(self.ref)) ** 2).sum()) / (self.S * self.N)

    def n3_max(self, rho):
        f = sum(4 * math.pi * R ** 3 * self.j3[i] * self.fwd(rho[i]) for i, R in enumerate(self.R))
        return float(self.inv(f).max())

    def picard(self, rho, V, iters, alpha, tol=0.0):
        """(rho, the last alpha, r before the last step) of the line-searched iteration."""
        g = self.G(rho, V)
        f0, prev, before = self.resid2(rho, g), 0.5, 0.0
        for _ in range(iters):
            if math.sqrt(f0) < tol:
                break
            m0, m1 = self.n3_max(rho), self.n3_max(g)
            top = min(1.0, (0.9 - m0) / (m1 - m0)) if m1 > m0 else 1.0
            if alpha >= 0:
                a = min(alpha, top)
            else:
                s = min(top, 2 * prev)
                mix = [(1 - t) * rho + t * g for t in (0.5 * s, s)]
                f1, f2 = (self.resid2(m, self.G(m, V)) for m in mix)
                c2, c1 = (f0 - 2 * f1 + f2) / (0.5 * s * s), (-3 * f0 + 4 * f1 - f2) / s
                a = min(max(-c1 / (2 * c2), 1e-3 * s), s) if c2 > 0 else (0.5 * s if f1 <= f2 else s)
            before, prev = math.sqrt(f0), a
            rho = (1 - a) * rho + a * g
            g = self.G(rho, V)
            f0 = self.resid2(rho, g)
        return rho, prev, before

    def fixed_point(self, rho, V, tol):
        """G(rho) = rho by Anderson mixing of log rho on the accessible voxels."""
        free = ~torch.isinf(V)
        u, us, fs = torch.log(rho[free]), [], []
        for it in range(600):
            x = torch.zeros_like(V)
            x[free] = torch.exp(u)
            g = self.G(x, V)
            if math.sqrt(self.resid2(x, g)) < tol:
                return x
            f = (torch.log(g[free]) - u).clamp(-1, 1)
            us, fs = (us + [u])[-9:], (fs + [f])[-9:]
            u = u + 0.1 * f
            if len(fs) > 1:
                A = torch.stack([b - a for a, b in zip(fs, fs[1:])], 1)
                X = torch.stack([b - a for a, b in zip(us, us[1:])], 1)
                y = torch.linalg.lstsq(A.cpu(), f[:, None].cpu(), driver="gelsd").solution.to(A.device)
                u = u - ((X + 0.1 * A) @ y)[:, 0]
        return None

    def omega(self, rho, V):
        free = ~torch.isinf(V) & (rho > 0)
        lr = torch.log(torch.where(free, rho, torch.ones_like(rho)) / self._col(self.rho_b))
        ext = torch.where(free, V, torch.zeros_like(V)) - self._col(self.mu_hs + self.mu_es)
        E, psi = self.screening(rho)
        drho = rho - self._col(self.rho_b)
        q = (self._col(self.z) * rho).sum(0)
        return self.dv * float((rho * (lr - 1 + ext) * free).sum() + _phi(self.weighted(rho), self.kind, "value").sum()
                               + 0.5 * (q * psi).sum() + (self._col(self.mu_es) * drho).sum() - 0.5 * (drho * E).sum())


def exact(case, seed):
    if case["op"] == "batch":
        got = []
        for i, m in enumerate(_members(case, seed)):
            dtype = torch.float64 if m["precision"] == "fp64" else torch.float32
            rho, V = (t.to(dtype).double() for t in _inputs(m, seed * 101 + i))
            got.append(_Exact(m).picard(rho, V, m["iters"], m["alpha"])[0])
        return {"rho": got}
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    rho, V = (t.to(dtype).double() for t in _inputs(case, seed))
    e = _Exact(case)
    op = case["op"]
    if op == "map":
        return {"G": e.G(rho, V)}
    if op == "fields":
        n = e.weighted(rho)
        E, psi = e.screening(rho)
        return {"n": n, "c1_hs": e.c1_hs(n), "c1_es": E - e._col(e.mu_es) - e._col(e.z) * psi, "psi": psi}
    if op == "grad":
        g = e.G(rho, V)
        ok = (rho > 0) & ~torch.isinf(V)
        d_rho = torch.where(ok, e.dv * torch.log(torch.where(ok, rho / g, torch.ones_like(rho))), torch.zeros_like(rho))
        d_bath = []
        for k in range(e.S):
            est = []
            for step in (1e-3, 5e-4):                   # central differences over the bath, extrapolated
                up, down = (e.molar * (1 + sign * step * (np.arange(e.S) == k)) for sign in (1, -1))
                est.append((_Exact(case, up).omega(rho, V) - _Exact(case, down).omega(rho, V)) / (2 * step * e.molar[k] * PER_NM3))
            d_bath.append((4 * est[1] - est[0]) / 3)
        return {"omega": torch.tensor(e.omega(rho, V), dtype=torch.float64), "d_rho": d_rho, "d_V": e.dv * rho,
                "d_bath": torch.tensor(d_bath, dtype=torch.float64)}
    if op == "newton":
        x = e.fixed_point(rho, V, 1e-2 * case["tol"])
        return None if x is None else {"rho": x}
    x, a, before = e.picard(rho, V, 1 if op == "step_host" else case["iters"], case["alpha"], case.get("tol", 0.0))
    return {"rho": x, "resid": before, "alpha": a} if op == "step_host" else {"rho": x}
