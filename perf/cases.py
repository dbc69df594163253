"""Performance cases of the force solver: what a user's program asks of it.

Each case is one call of the Python binding's public entry points (fmm_solve,
fmm_solve_graph, fmm_solve_batch, fmm_solve_jerk, fmm_direct, fmm_timesteps,
fmm_hold) on seeded synthetic star clusters drawn on the GPU: Plummer spheres
in Henon units (Mukherjee et al. 2021, Sec. 3), equal or Kroupa masses. The
sizes, orders and tolerances are those of this repository's benchmark, tests
and tuning tables, or lie between them.
"""
import math

import numpy as np
import torch

import paper_2012_02207_gb300 as gb

DEV = "cuda"
RMAX = 20.0  # the truncation radius of the cluster models, in virial radii
# MAC tolerances near the tuned ones of each expansion order (mixed precision, RMS error below 1e-6)
EPS_OF = {6: 1e-8, 8: 1e-8, 10: 2.8e-8, 12: 3e-8, 14: 2e-8}


def listed():
    return [
        # the smallest solve of the paper's accuracy study, in the default precision: launches and latency
        {"name": "solve_mixed_4k", "kind": "solve", "n": 4096, "p": 8, "eps": 1e-7, "leaf": 64,
         "precision": "mixed", "masses": "equal", "soft": 0.0},
        # the same in plain FP64
        {"name": "solve_fp64_4k", "kind": "solve", "n": 4096, "p": 8, "eps": 1e-7, "leaf": 64,
         "precision": "fp64", "masses": "equal", "soft": 0.0},
        # a softened solve (Appendix B, softening 1/N) at an odd size with small leaves and Kroupa masses
        {"name": "solve_soft_30k", "kind": "solve", "n": 30001, "p": 6, "eps": 1e-6, "leaf": 16,
         "precision": "mixed", "masses": "kroupa", "soft": 1.0 / 30001},
        # the repeated solve of a time-stepping loop on fixed buffers: a captured graph, replayed
        {"name": "graph_mixed_64k", "kind": "graph", "n": 65536, "p": 10, "eps": 2e-8, "leaf": 64,
         "precision": "mixed", "masses": "kroupa", "soft": 0.0},
        # the plain FP64 solve at the size of the paper's eps x p study
        {"name": "solve_fp64_100k", "kind": "solve", "n": 100000, "p": 10, "eps": 1e-7, "leaf": 64,
         "precision": "fp64", "masses": "equal", "soft": 0.0},
        # the headline: 2^20 stars with Kroupa masses in mixed precision, RMS error below 1e-6
        {"name": "solve_mixed_1m", "kind": "solve", "n": 1 << 20, "p": 10, "eps": 2.8e-8, "leaf": 64,
         "precision": "mixed", "masses": "kroupa", "soft": 0.0},
        # the largest: a nucleus-like cluster of 2^23 stars around a central point mass
        {"name": "solve_nucleus_8m", "kind": "solve", "n": (1 << 23) + 1, "p": 12, "eps": 2e-8, "leaf": 64,
         "precision": "mixed", "masses": "nucleus", "soft": 0.0},
        # an ensemble of clusters of uneven size in one call (N log-uniform in [2^10, 2^17])
        {"name": "batch_64_clusters", "kind": "batch", "clusters": 64, "log2_lo": 10.0, "log2_hi": 17.0,
         "sizes_seed": 4, "p": 12, "eps": 3e-8, "leaf": 128, "precision": "mixed"},
        # accelerations and jerks for a Hermite integrator
        {"name": "jerk_mixed_120k", "kind": "jerk", "n": 120001, "p": 10, "eps": 2e-8, "leaf": 64,
         "precision": "mixed", "masses": "kroupa", "soft": 0.0},
        # the FP64 direct sum at a sample of the bodies: how force errors are measured
        {"name": "direct_8k_of_128k", "kind": "direct", "n": 131072, "targets": 8192, "masses": "kroupa",
         "soft": 0.0},
        # individual step sizes of every body (Appendix A)
        {"name": "timesteps_16k", "kind": "timesteps", "n": 16384},
        # one step of the HOLD integrator (Appendix A, N = 100, dt = 1/16, eta of Table 1)
        {"name": "hold_100", "kind": "hold", "n": 100},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["mixed", "mixed", "mixed", "fp64", "graph", "batch", "jerk", "direct", "timesteps", "hold"])
    masses = rng.choice(["equal", "kroupa"])
    if kind in ("mixed", "graph", "jerk"):
        p = rng.choice([6, 8, 10, 12, 14])
        n = _log_int(rng, 1000, {"mixed": 1500000, "graph": 300000, "jerk": 300000}[kind])
        soft = 1.0 / n if kind != "graph" and rng.random() < 0.25 else 0.0
        return {"kind": "solve" if kind == "mixed" else kind, "n": n, "p": p,
                "eps": EPS_OF[p] * rng.choice([1.0, 3.0, 10.0]), "leaf": rng.choice([16, 32, 64, 64, 128]),
                "precision": "mixed", "masses": masses, "soft": soft}
    if kind == "fp64":  # orders up to 20, the paper's production choice
        return {"kind": "solve", "n": _log_int(rng, 1000, 60000), "p": rng.choice([6, 8, 10, 12, 16, 20]),
                "eps": rng.choice([1e-8, 1e-7, 1e-6]), "leaf": rng.choice([32, 64, 128]), "precision": "fp64",
                "masses": masses, "soft": 0.0}
    if kind == "batch":
        p = rng.choice([8, 10, 12])
        return {"kind": "batch", "clusters": _log_int(rng, 2, 100), "log2_lo": 9.0, "log2_hi": rng.choice([13.0, 15.0]),
                "sizes_seed": rng.randrange(1 << 20), "p": p, "eps": EPS_OF[p], "leaf": rng.choice([32, 64, 128]), "precision": "mixed"}
    if kind == "direct":
        n = _log_int(rng, 1000, 300000)
        return {"kind": "direct", "n": n, "targets": min(n, _log_int(rng, 256, 16384)), "masses": masses, "soft": 0.0}
    if kind == "timesteps":
        return {"kind": "timesteps", "n": _log_int(rng, 500, 20000)}
    return {"kind": "hold", "n": _log_int(rng, 24, 160)}


# ---------------------------------------------------------------- inputs

def _plummer(n, gen, virial_radius=1.0, total=1.0):
    """Positions (n, 3), velocities (n, 3) of a Plummer sphere in Henon units, isotropic, FP64 on the GPU."""
    def u(k):
        return torch.rand(k, generator=gen, device=DEV, dtype=torch.float64)

    def directions(k):
        c = 2.0 * u(k) - 1.0
        phi = (2.0 * math.pi) * u(k)
        s = torch.sqrt((1.0 - c * c).clamp(min=0.0))
        return torch.stack([s * torch.cos(phi), s * torch.sin(phi), c], 1)

    a = 3.0 * math.pi / 16.0
    xmax = RMAX ** 3 / (RMAX * RMAX + a * a) ** 1.5
    r = a / torch.sqrt((xmax * (1.0 - u(n))) ** (-2.0 / 3.0) - 1.0)
    pos = r[:, None] * directions(n)
    # speeds: a fraction q of the escape speed with density q^2 (1 - q^2)^{7/2}, by the inverse of its tabulated CDF
    grid = torch.linspace(0.0, 1.0, 4097, device=DEV, dtype=torch.float64)
    cdf = torch.cumsum(grid ** 2 * (1.0 - grid ** 2) ** 3.5, 0)
    cdf = cdf / cdf[-1].clone()
    t = u(n)
    k = torch.searchsorted(cdf, t).clamp(1, 4096)
    w = (t - cdf[k - 1]) / (cdf[k] - cdf[k - 1]).clamp(min=1e-300)
    q = grid[k - 1] + w.clamp(0.0, 1.0) * (grid[k] - grid[k - 1])
    vel = (q * math.sqrt(2.0 * total) * (r * r + a * a) ** (-0.25))[:, None] * directions(n)
    pos = pos - pos.mean(0)
    vel = vel - vel.mean(0)
    return pos * virial_radius, vel / math.sqrt(virial_radius)


def _masses(n, kind, gen, total=1.0):
    if kind != "kroupa":
        return torch.full((n,), total / n, device=DEV, dtype=torch.float64)
    # Kroupa (2001): dN/dm ~ m^-1.3 on [0.08, 0.5], m^-2.3 on [0.5, 150]
    lo, mid, hi, a1, a2 = 0.08, 0.5, 150.0, 1.3, 2.3
    k2 = mid ** (a2 - a1)
    w1 = (mid ** (1 - a1) - lo ** (1 - a1)) / (1 - a1)
    w2 = k2 * (hi ** (1 - a2) - mid ** (1 - a2)) / (1 - a2)
    t = torch.rand(n, generator=gen, device=DEV, dtype=torch.float64) * (w1 + w2)
    m1 = (lo ** (1 - a1) + t.clamp(max=w1) * (1 - a1)) ** (1.0 / (1 - a1))
    m2 = (mid ** (1 - a2) + (t - w1).clamp(min=0.0) * (1 - a2) / k2) ** (1.0 / (1 - a2))
    m = torch.where(t < w1, m1, m2).clamp(lo, hi)
    return m * (total / m.sum())


def _offsets(case):
    """Offsets and virial radii of an ensemble's clusters (part of the case: the seed draws the stars)."""
    rng = np.random.Generator(np.random.PCG64(case["sizes_seed"]))
    sizes = np.floor(2.0 ** rng.uniform(case["log2_lo"], case["log2_hi"], case["clusters"])).astype(np.int64)
    return np.concatenate([[0], np.cumsum(sizes)]), rng.uniform(0.5, 2.0, case["clusters"])


def _bodies(case, seed):
    """Contiguous columns x, y, z, vx, vy, vz, m of the case's bodies."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    if case["kind"] == "batch":
        # one draw of all the stars, then each cluster scaled by its own virial radius and mass 1
        offs, radii = _offsets(case)
        n = int(offs[-1])
        pos, vel = _plummer(n, gen)
        sizes = torch.from_numpy(np.diff(offs)).to(DEV)
        pos = pos * torch.repeat_interleave(torch.from_numpy(radii).to(DEV), sizes)[:, None]
        m = 1.0 / torch.repeat_interleave(sizes, sizes).to(torch.float64)
    elif case.get("masses") == "nucleus":
        n = case["n"] - 1
        pos, vel = _plummer(n, gen, total=0.99)
        zero = torch.zeros(1, 3, device=DEV, dtype=torch.float64)
        pos, vel = torch.cat([pos, zero]), torch.cat([vel, zero])
        m = torch.cat([_masses(n, "equal", gen, 0.99), torch.full((1,), 0.01, device=DEV, dtype=torch.float64)])
    else:
        pos, vel = _plummer(case["n"], gen)
        m = _masses(case["n"], case.get("masses", "equal"), gen)
    return [pos[:, d].contiguous() for d in range(3)] + [vel[:, d].contiguous() for d in range(3)] + [m]


def _targets(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed + 7)
    return torch.randperm(case["n"], generator=gen, device=DEV)[:case["targets"]].contiguous()


def prepare(case, seed):
    x, y, z, vx, vy, vz, m = _bodies(case, seed)
    kind = case["kind"]
    s = {"kind": kind, "xyzm": (x, y, z, m)}
    if kind in ("solve", "graph", "batch", "jerk"):
        s["fmm"] = gb.FMM(p=case["p"], eps=case["eps"], leaf_size=case["leaf"], precision=case["precision"],
                          soft=case.get("soft", 0.0))
    else:
        s["fmm"] = gb.FMM(soft=case.get("soft", 0.0))
    if kind == "graph":  # a time-stepping program keeps its force buffers
        s["out"] = tuple(torch.empty_like(x) for _ in range(4))
    elif kind == "batch":
        s["offsets"] = _offsets(case)[0]
    elif kind == "direct":
        s["targets"] = _targets(case, seed)
    if kind in ("jerk", "timesteps", "hold"):
        s["v"] = (vx, vy, vz)
    return s


def run(s):
    kind, f = s["kind"], s["fmm"]
    x, y, z, m = s["xyzm"]
    if kind == "solve":
        return f.solve(x, y, z, m)
    if kind == "graph":
        return f.solve_graph(x, y, z, m, out=s["out"])
    if kind == "batch":
        return f.solve_batch(s["offsets"], x, y, z, m)
    if kind == "jerk":
        return f.solve_jerk(x, y, z, *s["v"], m)
    if kind == "direct":
        return f.direct(x, y, z, m, targets=s["targets"])
    if kind == "timesteps":
        return f.timesteps(x, y, z, *s["v"], m, eta=0.025, symmetrize=True)
    # the integrator updates its bodies in place: each pass takes the same step from the same start
    w = [t.clone() for t in (x, y, z, *s["v"])]
    count = f.hold(*w, m, dt=1.0 / 16.0, nsteps=1, eta=0.025, symmetrize=True)
    return w, count


# ------------------------------------------------- the work of one pass

def work(case):
    """Bytes: inputs once and outputs once. Flops: 20 per body pair of a direct sum, 60 per pair of a symmetrized
    step size; for a solve, per body the near field of about twelve leaves each way (20 flops per mutual pair) and
    per leaf about 400 directed M2L of about 5 (p + 1)^3 flops (the lists at the tuned tolerances hold more)."""
    kind = case["kind"]
    n = int(_offsets(case)[0][-1]) if kind == "batch" else case["n"]
    if kind == "direct":
        return {"bytes": 32 * n + 40 * case["targets"], "flops": 20 * n * case["targets"]}
    if kind == "timesteps":
        return {"bytes": 64 * n, "flops": 60 * n * n}
    if kind == "hold":  # about 700 kicks and splits of sets of a third of the bodies, on the average
        return {"bytes": 104 * n, "flops": 80 * 700 * (n // 3) ** 2}
    leaf, p = case["leaf"], case["p"]
    near = 20 * n * min(n, 12 * leaf)
    far = (n / (0.5 * leaf)) * min(400, n / (0.5 * leaf)) * 5 * (p + 1) ** 3
    jerk = 2 if kind == "jerk" else 1
    return {"bytes": (32 + 32 + (48 if kind == "jerk" else 0)) * n, "flops": int(jerk * (near + far))}


# ------------------------------------------------ the same in 64 bits

def _chunks(n, k):
    step = max(1, min(n, (1 << 26) // k))
    return [(a, min(n, a + step)) for a in range(0, n, step)]


def _exact_forces(x, y, z, m, tgt, soft, v=None):
    """Direct sums at the targets: ax, ay, az, pot (and the jerk with velocities v)."""
    out = [torch.zeros(tgt.numel(), device=DEV, dtype=torch.float64) for _ in range(7 if v else 4)]
    for a, b in _chunks(tgt.numel(), x.numel()):
        i = tgt[a:b]
        d = [c[None, :] - c[i][:, None] for c in (x, y, z)]
        r2 = d[0] ** 2 + d[1] ** 2 + d[2] ** 2
        ri = torch.where(r2 > 0.0, r2 + soft * soft, torch.full_like(r2, math.inf)).rsqrt_()
        mr = m[None, :] * ri
        out[3][a:b] = -mr.sum(1)
        ri2 = ri * ri
        mr3 = mr * ri2
        for k in range(3):
            out[k][a:b] = (mr3 * d[k]).sum(1)
        if v:
            w = [c[None, :] - c[i][:, None] for c in v]
            rv3 = 3.0 * (d[0] * w[0] + d[1] * w[1] + d[2] * w[2]) * ri2
            for k in range(3):
                out[4 + k][a:b] = (mr3 * (w[k] - rv3 * d[k])).sum(1)
    return out


def _exact_steps(x, y, z, vx, vy, vz, m, eta):
    n = x.numel()
    tau = torch.empty_like(x)
    for a, b in _chunks(n, n):
        i = torch.arange(a, b, device=DEV)
        d = [c[None, :] - c[i][:, None] for c in (x, y, z)]
        w = [c[None, :] - c[i][:, None] for c in (vx, vy, vz)]
        gm = m[None, :] + m[i][:, None]
        r2, v2, rv = (sum(p * q for p, q in zip(s, t)) for s, t in ((d, d), (w, w), (d, w)))
        r = torch.sqrt(r2)
        tff = eta * torch.sqrt(r2 * r / gm)
        tfl = eta * r / torch.sqrt(v2)
        tff = tff / (1.0 - 0.5 * (1.5 * tff * rv / r2).clamp(max=1.0))
        tfl = tfl / (1.0 - 0.5 * (tfl * (rv / r2 + gm * rv / (r2 * r * v2))).clamp(max=1.0))
        t = torch.minimum(tff, tfl)
        t[i - a, i] = math.inf
        tau[a:b] = t.min(1).values
    return tau


def exact(case, seed):
    kind = case["kind"]
    if kind == "hold" or (kind != "batch" and case["n"] * case.get("targets", case["n"]) > 2 * 10 ** 10):
        return None  # a chaotic trajectory, or a direct sum that takes too long
    x, y, z, vx, vy, vz, m = _bodies(case, seed)
    if kind == "timesteps":
        return _exact_steps(x, y, z, vx, vy, vz, m, 0.025)
    soft = case.get("soft", 0.0)
    if kind == "batch":
        offs = _offsets(case)[0]
        if float((np.diff(offs).astype(np.float64) ** 2).sum()) > 4e10:
            return None
        parts = []
        for a, b in zip(offs[:-1], offs[1:]):
            parts.append(_exact_forces(*(c[a:b].contiguous() for c in (x, y, z, m)),
                                       torch.arange(int(b - a), device=DEV), soft))
        return [torch.cat(c) for c in zip(*parts)]
    tgt = _targets(case, seed) if kind == "direct" else torch.arange(case["n"], device=DEV)
    return _exact_forces(x, y, z, m, tgt, soft, (vx, vy, vz) if kind == "jerk" else None)
