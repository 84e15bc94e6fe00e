"""Performance cases of the directional FMM matvec: what users of the library have it do.

A case names a surface (points are made on the GPU from the seed), a tolerance, a number of
right-hand sides and the entry point the program calls:

  apply    u = G f on device buffers, plan resident (the call inside an iterative method)
  host     the same through host buffers: both copies and the wait are part of the call
  graph    the captured apply replayed on fixed device buffers
  batched  several geometries in one call (apply_batched)
  solve    restarted GMRES around the matvec

The tolerance picks the arithmetic: eps >= 1e-5 the tensor-core translations and the FP32 near field,
1e-6 the FP32 form, 1e-8 complex128 densities throughout.  Surfaces are sampled at about 100 points
per square wavelength (10 per wavelength), as the benchmark and the tests sample them.
"""
import math

import torch

from paper_1311_4257_gb300 import Plan, apply_batched

DENSITY = 100.0   # points per square wavelength


def listed():
    return [
        # the smallest call: a scatterer two wavelengths across; latency and launches count
        dict(name="sphere2", entry="apply", shape="sphere", K=2.0, n=1256, eps=1e-5, nrhs=1, leaf=64),
        # the tests' sphere of eight wavelengths at eps 1e-6, one right-hand side of a Krylov iteration
        dict(name="sphere8_1e-6", entry="apply", shape="sphere", K=8.0, n=20106, eps=1e-6, nrhs=1, leaf=64),
        # the benchmark's headline workload
        dict(name="sphere64_1e-5", entry="apply", shape="sphere", K=64.0, n=1286796, eps=1e-5, nrhs=1, leaf=64),
        # a large body at the tolerance between: FP32 arithmetic at scale
        dict(name="sphere32_1e-6", entry="apply", shape="sphere", K=32.0, n=321699, eps=1e-6, nrhs=1, leaf=64),
        # a group of sixteen incident fields on one body, as the request server forms them
        dict(name="ellipsoid32_rhs16", entry="apply", shape="ellipsoid", K=32.0, n=101247, eps=1e-5, nrhs=16, leaf=64),
        # a coarse survey of a ring-shaped body: low accuracy, an odd number of fields
        dict(name="torus40_1e-4_rhs3", entry="apply", shape="torus", K=40.0, n=252661, eps=1e-4, nrhs=3, leaf=64),
        # locally refined sampling: an adaptive low-frequency tree (leaves at several levels, W and X lists)
        dict(name="clustered8_leaf16", entry="apply", shape="clustered", K=8.0, n=20001, eps=1e-5, nrhs=1, leaf=16),
        # reference-quality potentials: complex128 densities at eps 1e-8
        dict(name="sphere8_1e-8", entry="apply", shape="sphere", K=8.0, n=20106, eps=1e-8, nrhs=1, leaf=64),
        # the same accuracy on a small body with edges and several fields
        dict(name="cube4_1e-8_rhs4", entry="apply", shape="cube", K=4.0, n=9600, eps=1e-8, nrhs=4, leaf=64),
        # four geometries of uneven size in one call, right-hand sides as in the batched benchmark
        dict(name="batch4", entry="batched", shape="mixed", K=16.0, n=80424, eps=1e-5, nrhs=32, leaf=64),
        # the solver: an integral equation of the second kind on a small body
        dict(name="solve4_1e-6", entry="solve", shape="sphere", K=4.0, n=5026, eps=1e-6, nrhs=1, leaf=64),
        # a program without device buffers: copies and the wait are part of the call
        dict(name="host16_1e-5", entry="host", shape="sphere", K=16.0, n=80424, eps=1e-5, nrhs=1, leaf=64),
    ]


def _surface(shape, K):
    """Area of the surface in square wavelengths, and its parameters."""
    if shape == "sphere" or shape == "clustered":
        return math.pi * K * K, ()
    if shape == "ellipsoid":   # semi-axes K/2, K/4, K/8 (Thomsen's approximation of the area)
        a, b, c, p = K / 2, K / 4, K / 8, 1.6075
        return 4 * math.pi * ((a ** p * b ** p + a ** p * c ** p + b ** p * c ** p) / 3) ** (1 / p), (a, b, c)
    if shape == "torus":       # radii R and R/4, K = 2.5 R
        R = K / 2.5
        return math.pi ** 2 * R * R, (R, R / 4)
    if shape == "cube":
        return 6 * K * K, ()
    raise ValueError(shape)


def draw(rng):
    """The listed cases' ranges: bodies of 2 to 48 wavelengths, 1 to 16 right-hand sides, every tolerance.
    The point count is the surface's at 100 per square wavelength, give or take a quarter."""
    eps = rng.choice([1e-3, 1e-4, 1e-5, 1e-5, 1e-6, 1e-6, 1e-8])
    entry = rng.choice(["apply", "apply", "apply", "apply", "graph", "host"])
    shape = rng.choice(["sphere", "sphere", "ellipsoid", "torus", "cube", "clustered"])
    top = 8.0 if eps < 1e-7 else 12.0 if shape == "clustered" else 32.0 if eps < 5e-6 else 48.0
    K = round(2.0 * (top / 2.0) ** rng.random(), 2)
    n = max(300, int(_surface(shape, K)[0] * DENSITY * rng.uniform(0.75, 1.25)))
    limit = 40_000 if eps < 1e-7 else 300_000 if eps < 5e-6 else 1_500_000   # points x right-hand sides
    n = min(n, limit)
    nrhs = rng.choice([k for k in (1, 1, 1, 2, 3, 4, 5, 7, 8, 16) if n * k <= limit])
    return dict(entry=entry, shape=shape, K=K, n=n, eps=eps, nrhs=nrhs, leaf=rng.choice([24, 64, 64, 100]))


# ---------------------------------------------------------------- inputs ---


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _unit(n, g):
    v = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
    return v / v.norm(dim=1, keepdim=True)


def _rand(g, *size):
    return torch.rand(*size, generator=g, device="cuda", dtype=torch.float64)


def _points(shape, K, n, seed):
    g = _gen(seed)
    if shape == "sphere":
        p = _unit(n, g) * (0.5 * K)
    elif shape == "ellipsoid":   # area-uniform by rejection from the unit sphere
        a, b, c = _surface(shape, K)[1]
        s = torch.tensor([a, b, c], device="cuda", dtype=torch.float64)
        got, have = [], 0
        while have < n:
            u = _unit(2 * n + 64, g)
            keep = _rand(g, u.shape[0]) < (u / s).norm(dim=1) * c
            got.append(u[keep] * s)
            have += got[-1].shape[0]
        p = torch.cat(got)[:n]
    elif shape == "torus":
        R, r = _surface(shape, K)[1]
        got, have = [], 0
        while have < n:
            t = _rand(g, 2 * n + 64) * (2 * math.pi)
            got.append(t[_rand(g, t.numel()) < (R + r * torch.cos(t)) / (R + r)])
            have += got[-1].numel()
        t = torch.cat(got)[:n]
        ph = _rand(g, n) * (2 * math.pi)
        q = R + r * torch.cos(t)
        p = torch.stack([q * torch.cos(ph), q * torch.sin(ph), r * torch.sin(t)], dim=1)
    elif shape == "cube":
        p = (_rand(g, n, 3) - 0.5) * K
        face = torch.randint(0, 6, (n,), generator=g, device="cuda")
        p[torch.arange(n, device="cuda"), face // 2] = torch.where(face % 2 == 0, 0.5 * K, -0.5 * K).to(torch.float64)
    elif shape == "clustered":   # a sphere with a third of its points in four tight clusters near it
        p = _unit(n, g) * (0.5 * K)
        c = _unit(4, g) * (0.45 * K)
        k = n // 3
        p[:k] = c[torch.randint(0, 4, (k,), generator=g, device="cuda")] + \
            0.05 * torch.randn(k, 3, generator=g, device="cuda", dtype=torch.float64)
    else:
        raise ValueError(shape)
    return p.clamp(-0.5 * K, 0.5 * K).contiguous()


def _densities(n, nrhs, dtype, seed):
    g = _gen(seed + 7919)
    real = torch.float64 if dtype == torch.complex128 else torch.float32
    return torch.view_as_complex(torch.randn(nrhs, n, 2, generator=g, device="cuda", dtype=real))


def _parts(case):
    """(shape, K, n, nrhs) of every geometry of the case: the batched one holds four, a quarter to one
    times the named size, with a growing number of right-hand sides."""
    if case["entry"] != "batched":
        return [(case["shape"], case["K"], case["n"], case["nrhs"])]
    K, n, r = case["K"], case["n"], case["nrhs"]
    return [("sphere", K / 2, n // 4 + 1, max(1, r // 32)), ("ellipsoid", K, 25312 * n // 80424, max(1, r // 8)),
            ("torus", 1.25 * K, 63165 * n // 80424, max(1, r // 2)), ("sphere", K, n, r)]


def _dtype(case):
    return torch.complex128 if case["eps"] < 1e-6 else torch.complex64


def _inputs(case, seed):
    return [(_points(s, K, n, seed + 1000 * i), K, _densities(n, r, _dtype(case), seed + 1000 * i))
            for i, (s, K, n, r) in enumerate(_parts(case))]


def _beta(case):
    # area per point / 4 pi, scaled by 4 / K so that the operator stays of the second kind as the body grows
    return _surface(case["shape"], case["K"])[0] / case["n"] / (4 * math.pi) * (4 / case["K"])


def prepare(case, seed):
    ins = _inputs(case, seed)
    plans = [Plan(p, K, case["eps"], leaf_max=case["leaf"]) for p, K, _ in ins]
    fs = [f for _, _, f in ins]
    st = dict(entry=case["entry"], plans=plans, fs=fs)
    if case["entry"] == "host":
        st["f_host"] = fs[0].cpu().pin_memory()
        st["u_host"] = torch.empty_like(st["f_host"]).pin_memory()
    elif case["entry"] == "graph":
        st["graph"] = plans[0].graph(fs[0], torch.empty_like(fs[0]))
    elif case["entry"] == "solve":
        st["beta"] = _beta(case)
    return st


def run(state):
    entry, plan, f = state["entry"], state["plans"][0], state["fs"][0]
    if entry == "apply":
        return plan.apply(f)
    if entry == "graph":
        return state["graph"].launch()
    if entry == "batched":
        return apply_batched(state["plans"], state["fs"])
    if entry == "host":
        plan.apply_host_ptr(state["f_host"].data_ptr(), state["u_host"].data_ptr(), f.shape[0])
        return state["u_host"]
    x, _, _ = plan.solve(f, alpha=1.0, beta=state["beta"], restart=30, maxit=30, tol=1e-6)
    return x


# translation flops per point and right-hand side (8 r_t r_s per box pair, unpadded ranks) on spheres,
# by tolerance: they change little with the size once there are high-frequency levels
TRANSLATION = {1e-3: 2.5e5, 1e-4: 3.8e5, 1e-5: 7.0e5, 1e-6: 1.1e6, 1e-8: 2.0e6}
NEAR = 260   # near-field interactions per point


def work(case):
    size = 16 if _dtype(case) == torch.complex128 else 8
    byt = flop = 0.0
    for _, _, n, r in _parts(case):
        byt += n * (24 + 2 * size * r)                                 # points, densities, potentials
        flop += n * r * TRANSLATION[case["eps"]] + n * NEAR * (16.0 + 8.0 * r)
    if case["entry"] == "solve":                                       # about fifteen matvecs to converge
        byt, flop = 15 * byt, 15 * flop
    return {"bytes": byt, "flops": flop}


# ----------------------------------------------------------------- exact ---


def _green(x, y):
    """exp(2 pi i d) / d between points x and y; coincident points give 0."""
    d2 = torch.zeros(x.shape[0], y.shape[0], device=x.device, dtype=torch.float64)
    for k in range(3):
        d2 += (x[:, k:k + 1] - y[None, :, k]) ** 2
    d = d2.sqrt_()
    inv = torch.where(d > 0, 1.0 / d, torch.zeros_like(d))
    return torch.polar(inv, (d - d.floor()) * (2 * math.pi))


def _direct(p, f):
    n = p.shape[0]
    u = torch.empty(n, f.shape[0], device="cuda", dtype=torch.complex128)
    ft = f.to(torch.complex128).T.contiguous()
    step = max(1, (1 << 27) // n)
    for i in range(0, n, step):
        u[i:i + step] = _green(p[i:i + step], p) @ ft
    return u.T.contiguous()


def exact(case, seed):
    """The direct sum of the kernel in 64 bits; the dense solve for the solver."""
    if sum(n * n * (150.0 + 8.0 * r) for _, _, n, r in _parts(case)) > 4e12:
        return None
    ins = _inputs(case, seed)
    if case["entry"] == "solve":
        p, _, b = ins[0]
        A = _green(p, p) * _beta(case) + torch.eye(p.shape[0], device="cuda", dtype=torch.complex128)
        return torch.linalg.solve(A, b.reshape(-1).to(torch.complex128))
    us = [_direct(p, f) for p, _, f in ins]
    if case["entry"] == "host":
        return us[0].cpu()
    return us if case["entry"] == "batched" else us[0]
