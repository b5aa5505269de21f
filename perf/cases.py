"""What this library is timed on: the long-range evaluations a discrete-element
or differentiable-simulation program asks it for, through the public API
(Plan, potential, field), from a few thousand particles to four million.

Inputs are drawn on the GPU from a seed: dense polydisperse packings (a
jittered lattice at solid fraction 0.4), uniform clouds, Plummer spheres,
rigid clumps and uneven batches, with the charges that go with them.  `exact`
is the direct O(N^2) sum (Ewald's sum in a periodic cell) in FP64.
"""
import math

import numpy as np
import torch

import paper_2512_09478_gb300 as kifmm

DEV = "cuda"
COULOMB = 1.0 / 8.8541878128e-12   # 1 / eps0, the SI coefficient of Eq. 3
GRAVITY = -4.0 * math.pi           # Eq. 4 with G = 1: attraction
MAX_PAIRS = 4.2e10                 # what exact() sums directly
KERNEL_FLOPS = 20                  # one pair: potential and gradient

DEFAULTS = dict(kind="forward", dist="packing", n=100_000, p=6, leaf=128, depth=20, precision="mixed_fp16",
                step="set", m2l_eps=0.0, systems=1, loss="")


def _case(name, **kw):
    c = dict(DEFAULTS, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the plain method on a small system in double precision: latency and launches
        _case("fp64_uniform_4096", dist="uniform", n=4096, p=4, leaf=64, precision="fp64"),
        # a small DEM run's step: as many launches as a large one, little work in each
        _case("dem_12k", n=12_345),
        # the headline: a million-sphere packing, tree rebuilt, potential and gradient
        _case("dem_1m", n=1_000_000),
        # rigid clumps of four charges: force and torque on each clump
        _case("clumps_200k", kind="clumps", dist="clumps", n=800_000),
        # a self-gravitating cloud: a deep adaptive tree at a high surface order
        _case("gravity_4m", dist="plummer", n=4_000_000, p=8, depth=12),
        # many independent systems of uneven size between tree rebuilds
        _case("batched_64", dist="batched", n=4_200_000, systems=64, leaf=64, step="update"),
        # single precision throughout, without the tensor-core split
        _case("fp32_dem_200k", n=200_003, precision="fp32"),
        # a converged reference field in double precision on a clustered cloud
        _case("fp64_plummer_60k", dist="plummer", n=60_001, leaf=64, precision="fp64"),
        # learning charges and positions from potentials: forward and backward
        _case("train_potential_130k", kind="train", loss="potential", n=130_001),
        # learning from forces: the adjoint of the gradient
        _case("train_forces_100k", kind="train", loss="forces", n=100_000),
        # a periodic cell of salt-like charges: forces and energy
        _case("periodic_120k", kind="periodic", dist="periodic", n=120_000),
        # suspended particles in Stokes flow: velocities from forces
        _case("stokes_60k", kind="stokes", dist="uniform", n=60_000, leaf=64, precision="fp32"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dem", "dem", "clumps", "gravity", "batched", "fp32", "fp64", "potential", "forces",
                       "periodic", "stokes"])
    if kind == "dem":
        return _case("", n=_logint(rng, 8_000, 1_000_000), p=rng.choice([4, 6, 6, 7]), leaf=rng.choice([64, 128]),
                     step=rng.choice(["set", "set", "update", "refresh"]), m2l_eps=rng.choice([0.0, 0.0, 0.0, 1e-5]))
    if kind == "clumps":
        return _case("", kind="clumps", dist="clumps", n=4 * _logint(rng, 5_000, 200_000),
                     step=rng.choice(["set", "update"]))
    if kind == "gravity":
        p = rng.choice([6, 8])
        return _case("", dist="plummer", n=_logint(rng, 30_000, 2_000_000), p=p, depth=12,
                     m2l_eps=rng.choice([0.0, 0.0, 1e-5]))
    if kind == "batched":
        s = _logint(rng, 4, 64)
        return _case("", dist="batched", n=s * _logint(rng, 8_000, 60_000), systems=s, leaf=64,
                     step=rng.choice(["set", "update"]))
    if kind == "fp32":
        return _case("", dist=rng.choice(["packing", "plummer", "uniform"]), n=_logint(rng, 5_000, 400_000),
                     p=rng.choice([4, 5, 6, 7]), leaf=rng.choice([64, 128]), precision="fp32")
    if kind == "fp64":
        return _case("", dist=rng.choice(["packing", "plummer", "uniform"]), n=_logint(rng, 2_000, 60_000),
                     p=rng.choice([4, 6, 6]), leaf=64, precision="fp64")
    if kind in ("potential", "forces"):
        prec = rng.choice(["mixed_fp16", "mixed_fp16", "fp32", "fp64"])
        return _case("", kind="train", loss=kind, dist=rng.choice(["packing", "plummer"]),
                     n=_logint(rng, 5_000, 10_000 if prec == "fp64" else 150_000), p=rng.choice([4, 6]),
                     leaf=rng.choice([64, 128]), precision=prec)
    if kind == "periodic":
        return _case("", kind="periodic", dist="periodic", n=2 * _logint(rng, 4_000, 75_000), p=rng.choice([4, 6]),
                     leaf=rng.choice([64, 128]), precision=rng.choice(["mixed_fp16", "fp32"]))
    prec = rng.choice(["fp32", "fp32", "fp64"])
    return _case("", kind="stokes", dist=rng.choice(["uniform", "packing"]),
                 n=_logint(rng, 2_000, 6_000 if prec == "fp64" else 60_000),
                 p=4 if prec == "fp64" else rng.choice([4, 6]), leaf=64, precision=prec)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _signs(g, n):
    return 2.0 * torch.randint(0, 2, (n,), generator=g, device=DEV).double() - 1.0


def _packing(g, n):
    """n sphere centres (mm) at solid fraction 0.4, radii about U[0.5, 1.5]: lattice cells jittered by
    +-0.28 of the spacing (no two centres closer than a small sphere's diameter), in random order."""
    m = int(math.ceil(n ** (1.0 / 3.0) - 1e-9))
    a = (4.0 / 3.0 * math.pi * 1.25 / 0.4) ** (1.0 / 3.0)
    cell = torch.randperm(m ** 3, generator=g, device=DEV)[:n]
    ijk = torch.stack([cell // (m * m), (cell // m) % m, cell % m], 1).double()
    return a * (ijk + 0.5 + 0.56 * (_rand(g, n, 3) - 0.5))


def _unit(g, n):
    d = _randn(g, n, 3)
    return d / d.norm(dim=1, keepdim=True)


def _plummer(g, n):
    """Plummer sphere of scale 1 cut at 20: radius by inverting M(<r) = r^3 / (r^2 + 1)^(3/2)."""
    top = 20.0 ** 3 / (20.0 ** 2 + 1.0) ** 1.5
    r = 1.0 / torch.sqrt((top * (_rand(g, n) * (1 - 1e-9) + 1e-9)) ** (-2.0 / 3.0) - 1.0)
    return _unit(g, n) * r[:, None]


def _sizes(systems, n):
    """Uneven system sizes adding up to n, log-uniform over a factor of 20 (a batch's layout stays, its particles move)."""
    w = np.exp(np.random.default_rng(17).uniform(0.0, math.log(20.0), systems))
    s = np.floor(n * w / w.sum()).astype(np.int64)
    s[-1] += n - s.sum()
    return s


def _inputs(case, seed):
    """positions, charges (or forces), system offsets, extra tensors; all FP64."""
    g, n, dist = _gen(seed), case["n"], case["dist"]
    extra = {}
    offsets = None
    if dist == "packing":
        x = _packing(g, n)
        q = 1e-12 * _randn(g, n)
    elif dist == "uniform":
        x = _rand(g, n, 3)
        q = _signs(g, n)
    elif dist == "plummer":
        x = _plummer(g, n)
        q = torch.exp(_randn(g, n))
    elif dist == "clumps":
        nc = n // 4
        side = 3.0 * nc ** (1.0 / 3.0)
        centres = side * _rand(g, nc, 3)
        body = _unit(g, n) * _rand(g, n, 1) ** (1.0 / 3.0)
        x = (centres[:, None, :] + body.view(nc, 4, 3)).reshape(-1, 3)
        q = 1e-12 * _randn(g, n)
        extra = {"centres": centres, "clump_offsets": 4 * torch.arange(nc + 1, device=DEV, dtype=torch.int64)}
    elif dist == "batched":
        sizes = _sizes(case["systems"], n)
        parts = [_rand(g, int(k), 3) if i % 2 == 0 else _plummer(g, int(k)) for i, k in enumerate(sizes)]
        x = torch.cat(parts)
        q = _signs(g, x.shape[0])
        offsets = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    elif dist == "periodic":
        x = _rand(g, n, 3)
        q = _signs(g, n // 2)
        q = torch.cat([q, -q])
    else:
        raise ValueError(dist)
    if case["kind"] == "stokes":
        q = _randn(g, n, 3)
    if case["kind"] == "train":
        extra = {"w": _randn(g, n), "g": _randn(g, n, 3)}
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    extra = {k: (v.to(dt) if v.is_floating_point() else v) for k, v in extra.items()}
    return x.to(dt), q.to(dt), offsets, extra


def _coef(case):
    if case["kind"] in ("stokes", "periodic", "train"):
        return 1.0
    return GRAVITY if case["dist"] == "plummer" else COULOMB if case["dist"] in ("packing", "clumps") else 1.0


def prepare(case, seed):
    x, q, offsets, extra = _inputs(case, seed)
    plan = kifmm.Plan(p=case["p"], leaf_cap=case["leaf"], max_depth=case["depth"], precision=case["precision"],
                      coef=_coef(case), n_max=x.shape[0], n_systems_max=case["systems"], dtype=x.dtype,
                      m2l_eps=case["m2l_eps"], cell=1.0 if case["kind"] == "periodic" else 0.0,
                      kernel="stokeslet" if case["kind"] == "stokes" else "laplace")
    if case["step"] != "set":
        plan.set_sources(x, q, offsets)  # the set-up's tree, kept between rebuilds
    return {"case": case, "plan": plan, "x": x, "q": q, "offsets": offsets, **extra}


def run(s):
    case, plan, x, q = s["case"], s["plan"], s["x"], s["q"]
    if case["kind"] == "train":
        xr, qr = x.detach().requires_grad_(), q.detach().requires_grad_()
        if case["loss"] == "potential":
            pot = kifmm.potential(xr, qr, plan)
            dx, dq = torch.autograd.grad(pot, (xr, qr), s["w"])
            return {"pot": pot.detach(), "dx": dx, "dq": dq}
        pot, grad = kifmm.field(xr, qr, plan)
        dx, dq = torch.autograd.grad(grad, (xr, qr), s["g"])
        return {"pot": pot.detach(), "grad": grad.detach(), "dx": dx, "dq": dq}
    if case["step"] == "update":
        plan.update_sources(x, q)
    elif case["step"] == "refresh":
        plan.refresh_sources(x, q)
    else:
        plan.set_sources(x, q, s["offsets"])
    if case["kind"] == "stokes":
        return {"velocity": plan.evaluate()[0]}
    if case["kind"] == "periodic":
        # what a time step needs: the potential's constant offset does not enter
        _, grad, energy = plan.evaluate(want_pot=False, want_energy=True)
        return {"grad": grad, "energy": energy}
    if case["kind"] == "clumps":
        pot, grad, _ = plan.evaluate()
        force, torque = plan.clump_reduce(s["clump_offsets"], x, q, grad, s["centres"])
        return {"pot": pot, "grad": grad, "force": force, "torque": torque}
    pot, grad, energy = plan.evaluate(want_energy=case["systems"] > 1)
    out = {"pot": pot, "grad": grad}
    if energy is not None:
        out["energy"] = energy
    return out


def work(case):
    """Inputs read once, outputs written once; the method's own arithmetic on an even cloud: pairs of
    adjacent leaves, surfaces of each leaf, one n_s x n_s translation per V-list entry."""
    n, p, leaf, S = case["n"], case["p"], case["leaf"], case["systems"]
    word = 8 if case["precision"] == "fp64" else 4
    comps = 3 if case["kind"] == "stokes" else 1
    values = 3 + comps + {"stokes": 3, "periodic": 3, "train": 4 + 4 + 4, "clumps": 4 + 3}.get(case["kind"], 4)
    ns = 6 * (p - 1) ** 2 + 2
    depth = max(0, math.ceil(math.log(max(1.0, n / S / leaf), 8)))
    leaves = S * 8 ** depth
    mean = min(leaf, n / leaves)
    boxes = leaves * 8 / 7 if depth else S
    near = n * (27 * mean + 2 * ns) * KERNEL_FLOPS * (comps + 1) / 2
    far = boxes * (189 * (min(1.0, depth / 3)) + 4) * 2 * (comps * ns) ** 2 if depth >= 2 else 0.0
    passes = {"potential": 2, "forces": 3}.get(case["loss"], 1)
    return {"bytes": float(values * word * n), "flops": float(passes * (near + far))}


# --------------------------------------------------------------------------
# the same outputs from the direct sums, FP64
# --------------------------------------------------------------------------
def _chunks(n, m):
    step = max(1, int(2 ** 26 // max(1, m)))
    for a in range(0, n, step):
        yield a, min(n, a + step)


def _direct(x, q, coef, w=None, g=None):
    """pot, grad of the charges q; with a loss sum w pot + sum g.grad also dq and dx.  FP64 [N]."""
    n = x.shape[0]
    k = coef / (4.0 * math.pi)
    pot, grad = torch.empty_like(q), torch.empty_like(x)
    dq, dx = (torch.zeros_like(q), torch.zeros_like(x)) if w is not None or g is not None else (None, None)
    for a, b in _chunks(n, n):
        r = [x[a:b, d, None] - x[None, :, d] for d in range(3)]
        r2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2]
        ri = torch.where(r2 > 0, r2, math.inf).rsqrt()
        ri3 = ri * ri * ri
        pot[a:b] = k * (ri @ q)
        f = [-k * ((r[d] * ri3) @ q) for d in range(3)]
        grad[a:b] = torch.stack(f, 1)
        if w is not None:
            dq[a:b] += k * (ri @ w)
            for d in range(3):
                dx[a:b, d] += w[a:b] * f[d] - q[a:b] * k * ((r[d] * ri3) @ w)
        if g is not None:
            ri5 = ri3 * ri * ri
            gr = sum(g[None, :, d] * r[d] for d in range(3))         # g_j . (x_i - x_j)
            dq[a:b] += k * (gr * ri3).sum(1)
            own = sum(g[a:b, d, None] * r[d] for d in range(3)) * ri5  # g_i . (x_i - x_j) / r^5
            mono = ri3 @ q
            for d in range(3):
                psi = ri3 @ g[:, d] - 3.0 * (gr * r[d] * ri5).sum(1)
                dx[a:b, d] += q[a:b] * k * psi + k * (3.0 * ((own * r[d]) @ q) - g[a:b, d] * mono)
    return pot, grad, dq, dx


def _stokes(x, f, coef):
    n = x.shape[0]
    v = torch.empty_like(x)
    for a, b in _chunks(n, n):
        r = [x[a:b, d, None] - x[None, :, d] for d in range(3)]
        r2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2]
        ri = torch.where(r2 > 0, r2, math.inf).rsqrt()
        rf = sum(r[d] * f[None, :, d] for d in range(3)) * (ri * ri * ri)
        for d in range(3):
            v[a:b, d] = ri @ f[:, d] + (rf * r[d]).sum(1)
    return coef / (8.0 * math.pi) * v


def _ewald_grad_energy(x, q, coef):
    """Gradient and energy of a neutral unit cell repeated over space (conducting boundary)."""
    n, alpha = x.shape[0], 11.0
    pot, grad = torch.zeros_like(q), torch.zeros_like(x)
    for a, b in _chunks(n, n):  # real space: nearest images (erfc(11 / 2) is about 7e-15)
        r = [x[a:b, d, None] - x[None, :, d] for d in range(3)]
        r = [t - torch.round(t) for t in r]
        r2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2]
        r2 = torch.where(r2 > 0, r2, math.inf)
        ri = r2.rsqrt()
        e = torch.special.erfc(alpha / ri) * ri
        e = torch.where(torch.isfinite(r2), e, 0.0)
        pot[a:b] = e @ q
        t = torch.where(torch.isfinite(r2), (e + 2 * alpha / math.sqrt(math.pi) * torch.exp(-alpha ** 2 * r2)) * ri * ri, 0.0)
        for d in range(3):
            grad[a:b, d] = -((r[d] * t) @ q)
    pot -= 2 * alpha / math.sqrt(math.pi) * q
    m = 20                                       # reciprocal space, half of the wave vectors
    k = torch.arange(-m, m + 1, device=DEV, dtype=torch.float64)
    K = torch.cartesian_prod(k, k, k)
    k2 = (K * K).sum(1)
    half = (K[:, 0] > 0) | ((K[:, 0] == 0) & ((K[:, 1] > 0) | ((K[:, 1] == 0) & (K[:, 2] > 0))))
    K, k2 = K[half & (k2 <= m * m)], k2[half & (k2 <= m * m)]
    amp = 2.0 / (math.pi * k2) * torch.exp(-math.pi ** 2 * k2 / alpha ** 2)
    for a, b in _chunks(K.shape[0], n):
        ph = 2 * math.pi * (x @ K[a:b].T)
        c, s = torch.cos(ph), torch.sin(ph)
        C, S = q @ c, q @ s
        pot += (c * (amp[a:b] * C) + s * (amp[a:b] * S)).sum(1)
        grad += 2 * math.pi * ((c * (amp[a:b] * S) - s * (amp[a:b] * C)) @ K[a:b])
    f = coef / (4 * math.pi)
    return f * grad, 0.5 * f * (q @ pot).reshape(1)


def exact(case, seed):
    x, q, offsets, extra = _inputs(case, seed)
    x, q = x.double(), q.double()
    coef = _coef(case)
    off = [0, x.shape[0]] if offsets is None else offsets.tolist()
    pairs = sum(float(b - a) ** 2 for a, b in zip(off[:-1], off[1:]))
    if pairs > MAX_PAIRS:
        return None
    if case["kind"] == "stokes":
        return {"velocity": _stokes(x, q, coef)}
    if case["kind"] == "periodic":
        grad, energy = _ewald_grad_energy(x, q, coef)
        return {"grad": grad, "energy": energy}
    if case["kind"] == "train":
        w = extra["w"].double() if case["loss"] == "potential" else None
        g = extra["g"].double() if case["loss"] == "forces" else None
        pot, grad, dq, dx = _direct(x, q, coef, w, g)
        out = {"pot": pot, "dx": dx, "dq": dq}
        return out if w is not None else dict(out, grad=grad)
    parts = [_direct(x[a:b], q[a:b], coef)[:2] for a, b in zip(off[:-1], off[1:])]
    pot, grad = torch.cat([t[0] for t in parts]), torch.cat([t[1] for t in parts])
    out = {"pot": pot, "grad": grad}
    if case["kind"] == "clumps":
        f = -(q[:, None] * grad)
        arm = x - extra["centres"].double().repeat_interleave(4, 0)
        out["force"] = f.view(-1, 4, 3).sum(1)
        out["torque"] = torch.linalg.cross(arm, f, dim=1).view(-1, 4, 3).sum(1)
    if case["systems"] > 1:
        out["energy"] = torch.stack([0.5 * (q[a:b] @ pot[a:b]) for a, b in zip(off[:-1], off[1:])])
    return out
