"""The solver calls whose time matters to users of this library, as measurable cases.

A case is one pass through a public entry point: a force evaluation (tg_fmm_forces), a rung-0 HOLD step
(tg_hhs_step), one step of an ensemble (tg_ensemble_step), direct summation for a sample of sinks
(tg_direct_forces) or the allocation-free Morton sort (tg_morton_sort_noalloc).  The particle sets are
those of paper_1712_10116_gb300/ics.py and of the benchmark's workloads, drawn here with torch on the GPU
so that a set of four million particles is ready in well under a second.  exact() evaluates the same
quantities by float64 direct summation in plain torch.

Case values: "do" the entry point, "dist" the particle set, "n" the particle count, "f64" the compute
precision (True: TG_PREC_FP64), "p" and "theta" the expansion order and opening angle, "n_crit" the leaf
size, "fast" the fraction of fast particles of a kick pair (0: every particle feels every mass), "pot"
whether the potential is asked for, "batched" the form of the HOLD step.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1712_10116_gb300 import ics
from paper_1712_10116_gb300 import binding as tg

# softening, its kernel and the integrator's settings of each particle set (the benchmark's workloads; the
# cube's softening follows the paper's scaling, the small clustered set's the tests')
SETS = {
    "plummer": dict(eps=0.01, kernel=tg.TG_KERNEL_PLUMMER, eta=0.025, dt_max=1.0 / 64, k_max=10),
    "sphere": dict(eps=0.005, kernel=tg.TG_KERNEL_WENDLAND_C2, eta=0.025, dt_max=1.0 / 16, k_max=10),
    "cube": dict(eps=0.01, kernel=tg.TG_KERNEL_WENDLAND_C2, eta=0.02, dt_max=1.0 / 64, k_max=10),
    "clustered": dict(eps=0.005, kernel=tg.TG_KERNEL_WENDLAND_C2, eta=0.025, dt_max=1.0 / 64, k_max=10),
    "disk": dict(eps=0.02, kernel=tg.TG_KERNEL_WENDLAND_C2, eta=0.025, dt_max=2.0, k_max=14),
}


def listed():
    return [
        # the smallest ensemble members evaluated alone: launches and host waits decide
        dict(name="eval_1k_f32", do="eval", dist="plummer", n=1021, f64=False, p=4, theta=0.5, n_crit=64, fast=0.0,
             pot=True),
        # the Plummer sphere of the float64 workload: its initial evaluation ...
        dict(name="eval_4k_f64", do="eval", dist="plummer", n=4096, f64=True, p=4, theta=0.5, n_crit=64, fast=0.0,
             pot=True),
        # ... and one of its rung-0 steps, as one graph launch
        dict(name="step_4k_f64", do="step", dist="plummer", n=4096, f64=True, p=4, theta=0.5, n_crit=64, batched=True),
        # the paper's cube collapse (momentum test) at the default parameters, host-driven step
        dict(name="step_cube_10k_f64", do="step", dist="cube", n=10000, f64=True, p=5, theta=0.45, n_crit=64,
             batched=False),
        # a kick pair of a mid-sized clustered system of odd size, at the paper's fiducial theta and p
        dict(name="kick_clustered_54k_f32", do="eval", dist="clustered", n=54321, f64=False, p=5, theta=0.45, n_crit=64,
             fast=0.3, pot=False),
        # the plain float64 path on an ordinary system, the reference of the float32 accuracy figures
        dict(name="kick_sphere_100k_f64", do="eval", dist="sphere", n=100003, f64=True, p=6, theta=0.5, n_crit=96,
             fast=0.3, pot=False),
        # the cold collapse: the evaluation that tg_hhs_init and every rung-0 kick do
        dict(name="eval_sphere_1m_f32", do="eval", dist="sphere", n=1 << 20, f64=False, p=6, theta=0.5, n_crit=96,
             fast=0.0, pot=False),
        # a kick pair of the disk galaxy, the largest force evaluation of the benchmark's headline step
        dict(name="kick_disk_4m_f32", do="eval", dist="disk", n=1 << 22, f64=False, p=6, theta=0.6, n_crit=96, fast=0.3,
             pot=False),
        # the benchmark's headline: one rung-0 step of the disk galaxy from t = 0, batched
        dict(name="step_disk_4m_f32", do="step", dist="disk", n=1 << 22, f64=False, p=6, theta=0.6, n_crit=128,
             batched=True),
        # independent systems stepped by one graph launch, each with its own rungs
        dict(name="ensemble_16_f32", do="ensemble", dist="plummer", systems=16, lo=1024, hi=32768, p=4, theta=0.5,
             n_crit=64),
        # the force-error gate: float64 direct summation for a sample of sinks
        dict(name="direct_4096_of_100k", do="direct", dist="sphere", n=100003, sinks=4096),
        # Morton keys and permutation for callers that must not allocate
        dict(name="sort_200k", do="sort", dist="clustered", n=200001),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: sizes spread over their logarithm, odd ones as likely as even ones."""
    do = rng.choices(["eval32", "eval64", "step32", "step64", "ensemble", "direct", "sort"], [6, 3, 3, 2, 1, 1, 1])[0]
    theta = rng.choice([0.45, 0.5, 0.6])
    p = rng.choice([4, 5, 6])
    n_crit = rng.choice([64, 96, 128])
    if do == "eval32":
        return dict(do="eval", dist=rng.choice(sorted(SETS)), n=_log_int(rng, 1000, 1 << 22), f64=False, p=p, theta=theta,
                    n_crit=n_crit, fast=rng.choice([0.0, 0.0, 0.1, 0.3, 0.7]), pot=rng.random() < 0.3)
    if do == "eval64":
        return dict(do="eval", dist=rng.choice(sorted(SETS)), n=_log_int(rng, 1000, 100000), f64=True, p=p, theta=theta,
                    n_crit=n_crit, fast=rng.choice([0.0, 0.3]), pot=rng.random() < 0.5)
    if do == "step32":
        return dict(do="step", dist=rng.choice(["plummer", "sphere", "disk"]), n=_log_int(rng, 2000, 1 << 20), f64=False,
                    p=p, theta=theta, n_crit=n_crit, batched=rng.random() < 0.7)
    if do == "step64":
        return dict(do="step", dist=rng.choice(["plummer", "cube"]), n=_log_int(rng, 1000, 16384), f64=True, p=p,
                    theta=theta, n_crit=64, batched=rng.random() < 0.5)
    if do == "ensemble":
        return dict(do="ensemble", dist="plummer", systems=rng.randint(4, 16), lo=1024, hi=_log_int(rng, 4096, 32768),
                    p=rng.choice([4, 5]), theta=theta, n_crit=n_crit)
    if do == "direct":
        return dict(do="direct", dist=rng.choice(["sphere", "plummer"]), n=_log_int(rng, 10000, 100000),
                    sinks=_log_int(rng, 64, 8192))
    return dict(do="sort", dist=rng.choice(["clustered", "sphere"]), n=_log_int(rng, 1000, tg.TG_NOALLOC_MAX_N))


# ------------------------------------------------------------------ particle sets
def _uniform(g, *shape):
    """Uniform draws in (0, 1), never 0."""
    return (torch.rand(*shape, generator=g, dtype=torch.float64, device="cuda") * (1 - 2.0 ** -52)) + 2.0 ** -53


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, dtype=torch.float64, device="cuda")


def _isotropic(g, n):
    c = 2.0 * _uniform(g, n) - 1.0
    phi = 2.0 * math.pi * _uniform(g, n)
    s = torch.sqrt(1.0 - c * c)
    return torch.stack([s * torch.cos(phi), s * torch.sin(phi), c])


def _plummer(g, n):
    """Plummer sphere (a = 1) inside r = 50; squared speeds in units of the escape speed follow
    q^2 (1 - q^2)^(7/2) dq, that is q^2 ~ Beta(3/2, 9/2), made of sums of squared normals."""
    x = _uniform(g, n) * (50.0 ** 3 / (1.0 + 2500.0) ** 1.5)
    r = 1.0 / torch.sqrt(x ** (-2.0 / 3.0) - 1.0)
    a, b = (_normal(g, 3, n) ** 2).sum(0), (_normal(g, 9, n) ** 2).sum(0)
    v = torch.sqrt(a / (a + b)) * math.sqrt(2.0) * (1.0 + r * r) ** -0.25
    return _isotropic(g, n) * r, _isotropic(g, n) * v


def _clustered(g, n):
    """Eight Plummer-like clumps on a uniform background, as ics.clustered."""
    nb = int(0.3 * n)
    centres = 0.8 * _uniform(g, 3, 8) - 0.4
    which = torch.randint(0, 8, (n - nb,), generator=g, device="cuda")
    x = (_uniform(g, n - nb)).clamp(1e-12, 1.0 - 1e-9)
    r = (0.05 / torch.sqrt(x ** (-2.0 / 3.0) - 1.0)).clamp(max=0.5)
    pos = torch.cat([centres[:, which] + _isotropic(g, n - nb) * r, _uniform(g, 3, nb) - 0.5], dim=1)
    return pos, 0.1 * _normal(g, 3, n)


def _interp(x, grid, values):
    """Piecewise linear interpolation of a table over a logarithmic grid."""
    lg = torch.log(torch.as_tensor(grid, device="cuda"))
    v = torch.as_tensor(values, device="cuda")
    t = torch.log(x.clamp(min=float(grid[0]), max=float(grid[-1])))
    i = torch.searchsorted(lg, t).clamp(1, lg.numel() - 1)
    w = (t - lg[i - 1]) / (lg[i] - lg[i - 1])
    return v[i - 1] * (1 - w) + v[i] * w


def _disk(g, n):
    """The disk galaxy of ics.disk_galaxy (exponential disk, Hernquist bulge, NFW halo) with velocities of
    the same Jeans moments, read from tables of ics.DiskGalaxyModel."""
    nd, nb = int(round(0.10 * n)), int(round(0.05 * n))
    nh = n - nd - nb
    model = ics.DiskGalaxyModel()
    R = -3.0 * torch.log(_uniform(g, nd) * _uniform(g, nd))
    phi = 2.0 * math.pi * _uniform(g, nd)
    c, s = torch.cos(phi), torch.sin(phi)
    disk = torch.stack([R * c, R * s, 0.3 * torch.atanh((2.0 * _uniform(g, nd) - 1.0) * (1.0 - 1e-12))])
    q = torch.sqrt(0.999 * _uniform(g, nb))
    bulge = _isotropic(g, nb) * (0.6 * q / (1.0 - q))
    x = np.geomspace(1e-6, 10.0, 8192)   # the NFW profile's enclosed mass, inverted from a table
    m = np.log1p(x) - x / (1.0 + x)
    u = _uniform(g, nh) * float(m[-1])
    halo = _isotropic(g, nh) * (3.0 * torch.exp(_interp(u, m, np.log(x))))
    grid = np.geomspace(1e-3, 60.0, 2048)
    sR2, sp2, sz2, vphi = (_interp(R, grid, t) for t in model.disk_moments(grid))
    vR, vp = _normal(g, nd) * torch.sqrt(sR2), vphi + _normal(g, nd) * torch.sqrt(sp2)
    vel = [torch.stack([vR * c - vp * s, vR * s + vp * c, _normal(g, nd) * torch.sqrt(sz2)])]
    for name, x3 in (("bulge", bulge), ("halo", halo)):
        rg = np.geomspace(1e-4, 40.0 if name == "halo" else 1300.0, 2048)
        sig = torch.sqrt(_interp(torch.linalg.norm(x3, dim=0), rg, model.sigma_r2(name, rg)))
        vel.append(_normal(g, 3, x3.shape[1]) * sig)
    mass = torch.cat([torch.full((k,), f / max(k, 1), dtype=torch.float64, device="cuda")
                      for k, f in ((nd, 0.10), (nb, 0.05), (nh, 0.85))])
    return torch.cat([disk, bulge, halo], dim=1), torch.cat(vel, dim=1), mass


def _particles(dist, n, seed):
    """(pos (3, n), vel (3, n), mass (n,)) float64 on the GPU, in a random order, total mass 1."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    mass = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
    if dist == "plummer":
        pos, vel = _plummer(g, n)
    elif dist == "sphere":
        pos = _isotropic(g, n) * _uniform(g, n) ** (1.0 / 3.0)
        vel = torch.zeros_like(pos)
    elif dist == "cube":
        pos = _uniform(g, 3, n) - 0.5
        vel = torch.zeros_like(pos)
    elif dist == "clustered":
        pos, vel = _clustered(g, n)
    else:
        pos, vel, mass = _disk(g, n)
    perm = torch.randperm(n, generator=g, device="cuda")
    return pos[:, perm].contiguous(), vel[:, perm].contiguous(), mass[perm].contiguous()


def _params(case):
    s = dict(SETS[case["dist"]])
    if case["dist"] == "cube":
        s["eps"] = ics.cube_softening(case["n"])
    if case["do"] == "direct":
        return tg.Params(precision=tg.TG_PREC_FP64, **s)
    f64 = case.get("f64", False)
    return tg.Params(p=case["p"], theta=case["theta"], n_crit=case["n_crit"],
                     precision=tg.TG_PREC_FP64 if f64 else tg.TG_PREC_FP32, batched=int(case.get("batched", False)), **s)


def _members(case, seed):
    """Sizes and seeds of an ensemble: sizes spread over their logarithm between lo and hi, both included,
    the same for every seed (the work of a case does not depend on the seed)."""
    k = case["systems"]
    ratio = case["hi"] / case["lo"]
    return [(int(round(case["lo"] * ratio ** (i / max(k - 1, 1)))), seed * 1000 + i) for i in range(k)]


def _fast_mask(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 7)
    return (torch.rand(case["n"], generator=g, device="cuda") < case["fast"]).to(torch.uint8)


# ------------------------------------------------------------------ prepare and run
class _Bound:
    """A system bound to a solver, with the state a pass starts from."""

    def __init__(self, params, pos, vel, mass):
        self.pos0, self.vel0, self.mass = pos, vel, mass
        self.pos, self.vel = pos.clone(), vel.clone()
        self.solver = tg.Solver(params)
        self.solver.hhs_init(self.pos, self.vel, self.mass)
        _, self.a_old, self.a_cur, self.a_tot = tg.tg_hhs_state(self.solver.ctx, mass.shape[0], with_total=True)

    def rewind(self):
        self.pos.copy_(self.pos0)
        self.vel.copy_(self.vel0)
        tg.tg_hhs_set_accel(self.solver.ctx, self.a_old, self.a_cur, self.a_tot)


def prepare(case, seed):
    if case["do"] == "ensemble":
        params = _params(dict(case, batched=True))
        return case, [_Bound(params, *_particles(case["dist"], n, s)) for n, s in _members(case, seed)]
    pos, vel, mass = _particles(case["dist"], case["n"], seed)
    if case["do"] == "step":
        return case, _Bound(_params(case), pos, vel, mass)
    if case["do"] == "sort":
        return case, (pos,)
    solver = tg.Solver(_params(case))
    if case["do"] == "direct":
        return case, (solver, pos, mass, torch.randperm(case["n"], device="cuda", generator=torch.Generator(
            device="cuda").manual_seed(seed + 11))[:case["sinks"]].contiguous())
    return case, (solver, pos, mass, _fast_mask(case, seed) if case["fast"] else None)


def run(state):
    case, s = state
    if case["do"] == "eval":
        solver, pos, mass, fast = s
        acc, pot = solver.fmm_forces(pos, mass, fast, want_pot=case["pot"])
        return {"acc": acc, "pot": pot} if case["pot"] else {"acc": acc}
    if case["do"] == "step":
        s.rewind()
        s.solver.hhs_step()
        return {"pos": s.pos, "vel": s.vel}
    if case["do"] == "ensemble":
        for b in s:
            b.rewind()
        tg.tg_ensemble_step([b.solver.ctx for b in s])
        return [{"pos": b.pos, "vel": b.vel} for b in s]
    if case["do"] == "direct":
        solver, pos, mass, sinks = s
        acc, pot = solver.direct_forces(pos, mass, None, sinks)
        return {"acc": acc, "pot": pot}
    keys, perm = tg.tg_morton_sort_noalloc(s[0])
    return {"keys": keys, "perm": perm}


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    """Inputs read once, outputs written once; flops of the method from the sizes alone.

    An evaluation meets a near field of the leaves within 2/theta sides (a leaf holds about a third of
    n_crit), each unordered pair once, 25 flops for both accelerations; about 500 cell pairs meet a cell in
    the far field (fewer where the tree is small), 4 (p+1)^4 / 3 flops each for both directions.  A HOLD step
    counts its set's particle-forces at t = 0 in units of n.  The direct sum takes 22 flops per pair."""
    if case["do"] == "sort":
        return {"bytes": 24.0 * case["n"] + 16.0 * case["n"], "flops": 0.0}
    if case["do"] == "direct":
        return {"bytes": 32.0 * case["n"] + 40.0 * case["sinks"], "flops": 22.0 * case["n"] * case["sinks"]}
    if case["do"] == "ensemble":
        each = [work(dict(case, do="step", n=n, batched=True)) for n, _ in _members(case, 0)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    n = float(case["n"])
    occ = case["n_crit"] / 3.0
    near = min(n / 2, 4.2 * (2.0 / case["theta"]) ** 3 * occ / 2)
    cells = n / occ
    far = min(cells / 8, 500.0) * cells * 4.0 * (case["p"] + 1) ** 4 / 3.0
    flops = n * near * 25.0 + far
    if case["do"] == "step":
        evals = {"plummer": 2.0, "sphere": 20.0, "cube": 6.0, "disk": 45.0}[case["dist"]]
        return {"bytes": 56.0 * n + 48.0 * n, "flops": evals * flops}
    out = 24.0 + (8.0 if case["pot"] else 0.0)
    return {"bytes": (32.0 + (1.0 if case["fast"] else 0.0) + out) * n, "flops": flops}


# ------------------------------------------------------------------ float64 by direct summation
PAIRS_MOST = 4e11   # directed pairs that plain torch sums in a few seconds


def _pair_values(r2, kernel, eps):
    """(g, phi) of a unit mass at squared distance r2: the force on a sink is g * (source - sink)."""
    if kernel == tg.TG_KERNEL_PLUMMER:
        inv = 1.0 / torch.sqrt(r2 + eps * eps)
        return inv ** 3, -inv
    r = torch.sqrt(r2)
    u = r / eps
    inv = 1.0 / r.clamp(min=eps)
    g = torch.where(u < 1, ((((21 * u - 90) * u + 140) * u - 84) * u * u + 14) / eps ** 3, inv ** 3)
    phi = torch.where(u < 1, ((((((3 * u - 15) * u + 28) * u - 21) * u * u + 7) * u * u) - 3) / eps, -inv)
    return g, phi


def _direct(pos, mass, kernel, eps, sinks, sources, drop=None, pot=False):
    """Accelerations (and potentials) of the sinks (indices) from the sources (indices), self excluded;
    drop (bool per particle): pairs with both members marked are left out."""
    acc = torch.zeros(3, sinks.numel(), dtype=torch.float64, device="cuda")
    phi = torch.zeros(sinks.numel(), dtype=torch.float64, device="cuda")
    xs, ms = pos[:, sources], mass[sources]
    step = max(1, (1 << 25) // max(1, sources.numel()))
    for i in range(0, sinks.numel(), step):
        t = sinks[i:i + step]
        d = [xs[k][None, :] - pos[k, t][:, None] for k in range(3)]
        g, ph = _pair_values(d[0] * d[0] + d[1] * d[1] + d[2] * d[2], kernel, eps)
        w = ms[None, :] * (t[:, None] != sources[None, :])
        if drop is not None:
            w = w * ~(drop[t][:, None] & drop[sources][None, :])
        g = g * w
        for k in range(3):
            acc[k, i:i + step] = (g * d[k]).sum(1)
        if pot:
            phi[i:i + step] = (ph * w).sum(1)
    return acc, phi


def _hold_step(prm, pos, vel, mass):
    """One rung-0 step of EVOLVE_HOLD by direct summation (the paper's Algorithms 1-3)."""
    n = mass.numel()
    everyone = torch.arange(n, device="cuda")
    force = lambda sinks, sources: _direct(pos, mass, prm.kernel, prm.eps, sinks, sources)[0]  # noqa: E731
    a_old = torch.zeros(n, dtype=torch.float64, device="cuda")
    a_cur = torch.linalg.norm(force(everyone, everyone), dim=0)
    dts = torch.zeros_like(a_old)
    spent = [0]

    def kick(S, F, dt, second):
        spent[0] += S.numel() * (S.numel() + 2 * F.numel())
        if spent[0] > PAIRS_MOST:
            raise OverflowError
        a_s = force(S, torch.cat([S, F]))
        a_f = force(F, S) if F.numel() else None
        vel[:, S] += a_s * (0.5 * dt)
        a_cur[S] = torch.linalg.norm(a_s, dim=0)
        if F.numel():
            vel[:, F] += a_f * (0.5 * dt)
            if second:
                a_old[F] = torch.linalg.norm(a_f, dim=0)

    def evolve(k, idx, dt, calc):
        if calc:
            dts[idx] = torch.sqrt(prm.eta * prm.eps / (a_old[idx] + a_cur[idx]))
        fast = dts[idx] < dt if k < prm.k_max else torch.zeros_like(idx, dtype=torch.bool)
        S, F = idx[~fast], idx[fast]
        if F.numel():
            evolve(k + 1, F, dt / 2, False)
        if S.numel():
            kick(S, F, dt, False)
            pos[:, S] += vel[:, S] * dt
            kick(S, F, dt, True)
        if F.numel():
            evolve(k + 1, F, dt / 2, True)

    evolve(0, everyone, prm.dt_max, True)
    return {"pos": pos, "vel": vel}


def exact(case, seed):
    """The outputs of run() for these inputs from float64 direct summation, or None where that takes long.
    Keys and permutations are whole numbers and have no such value."""
    if case["do"] == "sort" or case["do"] == "eval" and float(case["n"]) ** 2 > PAIRS_MOST:
        return None
    try:
        if case["do"] == "ensemble":
            if sum(12.0 * n * n for n, _ in _members(case, seed)) > PAIRS_MOST:
                return None
            return [_hold_step(_params(case), *_particles(case["dist"], n, s)) for n, s in _members(case, seed)]
        if case["do"] == "step" and 4.0 * float(case["n"]) ** 2 > PAIRS_MOST:
            return None
        pos, vel, mass = _particles(case["dist"], case["n"], seed)
        prm = _params(case)
        if case["do"] == "step":
            return _hold_step(prm, pos, vel, mass)
    except OverflowError:
        return None
    everyone = torch.arange(case["n"], device="cuda")
    if case["do"] == "direct":
        sinks = torch.randperm(case["n"], device="cuda", generator=torch.Generator(device="cuda").manual_seed(
            seed + 11))[:case["sinks"]]
        acc, phi = _direct(pos, mass, prm.kernel, prm.eps, sinks, everyone, pot=True)
        return {"acc": acc, "pot": phi}
    drop = _fast_mask(case, seed).bool() if case["fast"] else None
    acc, phi = _direct(pos, mass, prm.kernel, prm.eps, everyone, everyone, drop, case["pot"])
    return {"acc": acc, "pot": phi} if case["pot"] else {"acc": acc}
