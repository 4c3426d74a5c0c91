"""The calls whose speed is measured: what a program built on this package has
the GPU do, through the package's public entry points, over the sizes of the
repository's own configurations, tests and benchmark.

Inputs are drawn on the GPU from the seed alone, with the distributions of
workloads/ (jittered lattice; Gaussian blobs on a uniform background with
log-normal masses). exact() restates each path in 64-bit torch, by brute force
over the particles (and, for gravity, by a breadth-first walk of the tree that
include/sph.h defines), without this package's code.
"""
from __future__ import annotations

import math

import torch

GAMMA = 5.0 / 3.0
N_TARGET = 64.0
PAIRS_DENSITY = 60      # neighbours within h per particle (N_eff = 64 number-weighted)
PAIRS_FORCE = 80        # partners within max(h_i, h_j) per particle
FLOPS_DENSITY, FLOPS_FORCE, FLOPS_GRAVITY = 30, 90, 40   # per pair, node or particle interaction


def listed():
    return [
        # One step of a small box (the smoke test's lattice, the smallest of the batched
        # boxes): a few launches' worth of work, so latency and the number of launches.
        {"name": "step_lattice_4k", "kind": "step", "n": 4096, "shape": "lattice", "f64": False},
        # The plain method in double on the 32^3 lattice: FP64 positions and pair arithmetic,
        # the run that the FP32 results are checked against.
        {"name": "step_lattice_33k_f64", "kind": "step", "n": 32768, "shape": "lattice", "f64": True},
        # One step of a clustered box at an odd size: grid rebuild, density, force.
        {"name": "step_clustered_300k", "kind": "step", "n": 300_007, "shape": "clustered", "f64": False},
        # The benchmark's step: 10M clustered particles whose time bins give sub-steps with
        # 100, 10, 1 and 0.1 % active.
        {"name": "timebins_10m", "kind": "timebins", "n": 10_000_000, "fraction": 1.0},
        # A sparse sub-step of the 2M box, the usual tick of a run on time bins.
        {"name": "substep_2m_1pct", "kind": "substep", "n": 2_097_152, "fraction": 0.01},
        # Many small uneven boxes in one grid, one launch per pass.
        {"name": "boxes_64", "kind": "boxes", "boxes": 64, "n_min": 4096, "n_max": 65_536, "sizes": 4},
        # "Improved SPH": density with div v and curl v, force with Balsara's switch and a
        # viscosity parameter per particle, and its rate.
        {"name": "viscosity_262k", "kind": "viscosity", "n": 262_144, "fraction": 1.0},
        # The force pass with thermal conduction after a density pass that recorded the
        # neighbour lists.
        {"name": "conduction_800k", "kind": "conduction", "n": 800_003, "fraction": 1.0},
        # Short-range gravity of every particle, the split of a mesh of one cell per spacing.
        {"name": "gravity_1m", "kind": "gravity", "n": 1_000_000, "theta": 0.5, "fraction": 1.0},
        # The same for a sub-step's active particles of a small box.
        {"name": "gravity_30k_subset", "kind": "gravity", "n": 30_000, "theta": 0.5, "fraction": 0.3},
        # Forward and backward through the differentiable density and force.
        {"name": "adjoint_262k", "kind": "adjoint", "n": 262_144},
        # A dt_max cycle of the integrator: drift, rebuild, active sets, forces, kicks, bins.
        {"name": "kdk_cycle_66k", "kind": "kdk", "n": 65_537, "max_bin": 3},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "timebins", "substep", "boxes", "viscosity", "conduction", "gravity", "gravity",
                       "adjoint", "kdk"])
    frac = round(math.exp(rng.uniform(math.log(0.002), math.log(1.0))), 4)
    if kind == "step":
        f64 = rng.random() < 0.2
        shape = rng.choice(["lattice", "clustered"])
        n = _log(rng, 4096, 32_768 if f64 else 2_000_000)
        if shape == "lattice":
            n = max(16, round(n ** (1 / 3))) ** 3
        return {"kind": kind, "n": n, "shape": shape, "f64": f64}
    if kind == "timebins":
        return {"kind": kind, "n": _log(rng, 500_000, 8_000_000), "fraction": 1.0}
    if kind == "substep":
        return {"kind": kind, "n": _log(rng, 50_000, 4_000_000), "fraction": frac}
    if kind == "boxes":
        n_min = _log(rng, 2048, 16_384)
        return {"kind": kind, "boxes": rng.randint(3, 64), "n_min": n_min, "n_max": _log(rng, n_min, 131_072),
                "sizes": rng.randrange(1 << 20)}
    if kind == "viscosity":
        return {"kind": kind, "n": _log(rng, 30_000, 2_000_000), "fraction": rng.choice([1.0, frac])}
    if kind == "conduction":
        return {"kind": kind, "n": _log(rng, 30_000, 2_000_000), "fraction": rng.choice([1.0, frac])}
    if kind == "gravity":
        return {"kind": kind, "n": _log(rng, 10_000, 1_500_000), "theta": rng.choice([0.0, 0.3, 0.5, 0.7, 1.0]),
                "fraction": rng.choice([1.0, frac])}
    if kind == "adjoint":
        return {"kind": kind, "n": _log(rng, 10_000, 600_000)}
    return {"kind": "kdk", "n": _log(rng, 8192, 200_000), "max_bin": rng.randint(1, 3)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _rand(gen, *shape):
    return torch.rand(*shape, device="cuda", dtype=torch.float64, generator=gen)


def _randn(gen, *shape):
    return torch.randn(*shape, device="cuda", dtype=torch.float64, generator=gen)


def _wrap32(x):
    """FP64 positions rounded to FP32 and folded into [0, 1)."""
    x = x.remainder(1.0).float()
    return torch.where(x >= 1.0, torch.zeros_like(x), x)


def _lattice(n, gen):
    side = round(n ** (1 / 3))
    g = (torch.arange(side, device="cuda", dtype=torch.float64) + 0.5) / side
    pos = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    pos = pos + (0.6 * _rand(gen, n, 3) - 0.3) / side
    return dict(pos=pos.remainder(1.0), mass=torch.full((n,), 1.0 / n, device="cuda"),
                vel=(0.1 * _randn(gen, n, 3)).float(), u=(0.9 + 0.2 * _rand(gen, n)).float(),
                rank=torch.rand(n, device="cuda", generator=gen))


def _clustered(n, gen):
    """70 % of the particles in Gaussian blobs (sigma log-uniform in [0.002,
    0.05]), 30 % uniform. `rank` orders them as time steps do: compact and hot
    first."""
    blobs = max(1, round(0.158 * math.sqrt(n)))
    nb = round(0.7 * n)
    sig = torch.exp(math.log(0.002) + math.log(25.0) * _rand(gen, blobs))
    centre, bulk = _rand(gen, blobs, 3), 0.1 * _randn(gen, blobs, 3)
    member = torch.randint(blobs, (nb,), device="cuda", generator=gen)
    pos = torch.cat([centre[member] + _randn(gen, nb, 3) * sig[member, None], _rand(gen, n - nb, 3)])
    vel = 0.1 * _randn(gen, n, 3)
    vel[:nb] += bulk[member]
    mass = torch.exp(_randn(gen, n))
    u = 10.0 ** (2.0 * _rand(gen, n) - 1.0)
    rank = torch.full((n,), 0.1, device="cuda", dtype=torch.float64)
    rank[:nb] = sig[member]
    rank = rank / u.sqrt()
    order = torch.randperm(n, device="cuda", generator=gen)
    return dict(pos=pos.remainder(1.0)[order].contiguous(), mass=(mass / mass.sum()).float()[order].contiguous(),
                vel=vel.float()[order].contiguous(), u=u.float()[order].contiguous(), rank=rank[order].contiguous())


def _particles(case, gen):
    p = _lattice(case["n"], gen) if case.get("shape") == "lattice" else _clustered(case["n"], gen)
    if not case.get("f64"):
        p["pos"] = _wrap32(p["pos"])
    return p


def _box_sizes(case):
    g = torch.Generator().manual_seed(case["sizes"])
    r = torch.rand(case["boxes"], generator=g, dtype=torch.float64)
    lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
    return [int(round(math.exp(lo + (hi - lo) * float(v)))) for v in r]


def _boxes(case, gen):
    sizes = _box_sizes(case)
    parts = [_clustered(n, gen) for n in sizes]
    p = {k: torch.cat([q[k] for q in parts]).contiguous() for k in ("pos", "mass", "vel", "u")}
    p["pos"] = _wrap32(p["pos"])
    offs = [0]
    for n in sizes:
        offs.append(offs[-1] + n)
    return p, offs


def _morton_order(S, ctx, p, params):
    """The particles stored along the grid's curve, as a run keeps them."""
    grid = S.sph_build_grid(ctx, p["pos"], p["mass"], params)
    perm = torch.empty(p["pos"].shape[0], dtype=torch.int32, device="cuda")
    S.sph_grid_export(grid, perm)
    order = perm.long()
    p = {k: v[order].contiguous() for k, v in p.items()}
    grid.free()
    return p


def _first(p, fraction):
    """The caller indices of the `fraction` of the particles with the smallest time step."""
    n = p["pos"].shape[0]
    k = max(1, round(fraction * n))
    if k >= n:
        return None   # every particle
    return p["rank"].argsort(stable=True)[:k].sort().values.int()


def _gravity_split(n):
    cell = 1.0 / round(n ** (1 / 3))
    return dict(r_split=1.25 * cell, r_cut=min(4.5 * 1.25 * cell, 0.25), h_soft=2.8 * cell / 30)


def _seeds(n, gen):
    """dL/da and dL/drho of the adjoint."""
    return _randn(gen, n, 3).float(), _randn(gen, n).float()


def prepare(case, seed):
    import paper_2003_10850_gb300 as S

    kind, gen = case["kind"], _gen(seed)
    ctx = S.Context(0)
    params = S.default_params(flags=S.SPH_FP64 if case.get("f64") else 0)
    if kind == "boxes":
        p, offs = _boxes(case, gen)
    else:
        p, offs = _particles(case, gen), None
    if kind in ("timebins", "substep"):
        p = _morton_order(S, ctx, p, params)
    n = p["pos"].shape[0]
    st = {"S": S, "ctx": ctx, "params": params, "kind": kind, "n": n, "p": p}
    z = lambda *s: torch.zeros(*s, device="cuda")

    if kind == "adjoint":
        for k in ("pos", "mass", "u"):
            p[k].requires_grad_(True)
        st["h0"] = z(n)
        st["seeds"] = _seeds(n, gen)
        return st

    if kind == "kdk":
        # the finest bin holds the smallest Courant step, found from a density and a force pass
        from paper_2003_10850_gb300.kdk import KDK
        grid = S.sph_build_grid(ctx, p["pos"], p["mass"], params)
        h = z(n)
        d = S.density(ctx, grid, h, None, params)
        f = S.hydro_force(ctx, grid, p["vel"], p["u"], h, d["rho"], d["omega"], None, params)
        S.sph_sync_status(ctx)
        grid.free()
        dt_min = float((0.3 * h / f["vsig"].clamp_min(1e-30)).min())
        dt_max = float("%.2g" % (0.9 * 2 ** case["max_bin"] * dt_min))
        run = KDK(ctx, p["pos"].double(), p["mass"], p["vel"], p["u"], dt_max, case["max_bin"])
        st["kdk"] = run
        names = ("pos", "vel", "u", "vel_pred", "u_pred", "h", "rho", "omega", "acc", "dudt", "vsig", "bins")
        st["saved"] = {k: getattr(run, k).clone() for k in names}
        return st

    if offs is None:
        st["grid"] = S.sph_build_grid(ctx, p["pos"], p["mass"], params)
    else:
        st["grid"] = S.sph_build_grid_batched(ctx, p["pos"], p["mass"], offs, [1.0] * (len(offs) - 1), params)
    if kind == "gravity":
        st["gp"] = S.gravity_params(G=1.0, theta=case["theta"], **_gravity_split(n))
        st["active"] = _first(p, case["fraction"])
        st["acc"] = z(n, 3)
        st["n_nodes"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        st["n_pairs"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        return st

    st["h"] = z(n)
    st["rho"], st["omega"], st["acc"], st["dudt"], st["vsig"] = z(n), z(n), z(n, 3), z(n), z(n)
    st["n_ngb"] = torch.zeros(n, dtype=torch.int32, device="cuda")
    st["flags"] = torch.zeros(n, dtype=torch.uint8, device="cuda")
    # the smoothing lengths that a run carries from its last step: converged, then off by what
    # the density changes between two steps (2 %) on the particles that become active
    S.sph_density(ctx, st["grid"], st["h"], None, st["rho"], st["omega"], st["n_ngb"], st["flags"], None, params)
    S.sph_sync_status(ctx)
    scatter = torch.exp(0.02 * _randn(gen, n)).float()
    if kind == "timebins":
        st["sets"] = [_first(p, f) for f in (1.0, 0.1, 0.01, 0.001)]
    else:
        st["sets"] = [_first(p, case.get("fraction", 1.0))]
    st["guess"] = []
    for a in st["sets"]:
        g = st["h"].clone()
        if a is None:
            g *= scatter
        else:
            g[a.long()] *= scatter[a.long()]
        st["guess"].append(g)
    if kind == "viscosity":
        st["divv"], st["curlv"], st["dalpha"] = z(n), z(n), z(n)
        S.sph_density_divcurl(ctx, st["grid"], st["h"], None, st["rho"], st["omega"], st["n_ngb"], st["flags"], None,
                              p["vel"], st["divv"], st["curlv"], params)
        st["alpha"] = (0.1 + 0.9 * _rand(gen, n)).float()
    if kind == "conduction":
        st["kappa"] = (10.0 ** (_rand(gen, n) - 1.0)).float()
        st["dcond"] = z(n)
        st["h"].copy_(st["guess"][0])
        S.sph_density(ctx, st["grid"], st["h"], st["sets"][0], st["rho"], st["omega"], st["n_ngb"], st["flags"], None,
                      params)
    S.sph_sync_status(ctx)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(st):
    S, ctx, p, kind, params = st["S"], st["ctx"], st["p"], st["kind"], st["params"]
    if kind == "adjoint":
        from paper_2003_10850_gb300.autograd import SPHDensityForce
        acc, rho = SPHDensityForce.apply(p["pos"], p["vel"], p["mass"], p["u"], st["h0"], ctx, params)
        g = torch.autograd.grad((acc, rho), (p["pos"], p["mass"], p["u"]), st["seeds"])
        return {"acc": acc, "rho": rho, "g_pos": g[0], "g_mass": g[1], "g_u": g[2]}
    if kind == "kdk":
        k = st["kdk"]
        for name, v in st["saved"].items():
            getattr(k, name).copy_(v)
        k.tick = 0
        for _ in range(1 << k.max_bin):
            k.step(sync=False)
        return {name: getattr(k, name) for name in ("pos", "vel", "u", "h", "rho", "acc", "dudt", "vsig", "bins")}
    grid = st["grid"]
    if kind == "gravity":
        S.sph_gravity(ctx, grid, st["active"], st["gp"], st["acc"], st["n_nodes"], st["n_pairs"])
        return {k: st[k] for k in ("acc", "n_nodes", "n_pairs")}
    h, rho, omega, act = st["h"], st["rho"], st["omega"], st["sets"][0]
    if kind == "conduction":
        S.sph_hydro_force_conduction(ctx, grid, p["vel"], p["u"], h, rho, omega, None, None, st["kappa"], act,
                                     st["acc"], st["dudt"], st["vsig"], st["dcond"], None, params)
        return {k: st[k] for k in ("acc", "dudt", "vsig", "dcond")}
    if kind == "viscosity":
        h.copy_(st["guess"][0])
        S.sph_density_divcurl(ctx, grid, h, act, rho, omega, st["n_ngb"], st["flags"], None, p["vel"], st["divv"],
                              st["curlv"], params)
        S.sph_hydro_force_visc(ctx, grid, p["vel"], p["u"], h, rho, omega, st["alpha"], st["divv"], st["curlv"], act,
                               st["acc"], st["dudt"], st["vsig"], None, params)
        S.sph_visc_rate(ctx, act, h, p["u"], st["divv"], st["alpha"], st["dalpha"])
        return {k: st[k] for k in ("h", "rho", "omega", "n_ngb", "flags", "divv", "curlv", "acc", "dudt", "vsig",
                                   "dalpha")}
    if kind != "substep":
        S.sph_grid_update(ctx, grid, p["pos"], p["mass"])
    for act, guess in zip(st["sets"], st["guess"]):
        h.copy_(guess)
        S.sph_density(ctx, grid, h, act, rho, omega, st["n_ngb"], st["flags"], None, params)
        S.sph_hydro_force(ctx, grid, p["vel"], p["u"], h, rho, omega, act, st["acc"], st["dudt"], st["vsig"], None,
                          params)
    return {k: st[k] for k in ("h", "rho", "omega", "n_ngb", "flags", "acc", "dudt", "vsig")}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Inputs read once, outputs written once (per active particle where only
    those are needed); flops of the pairs at the converged h, evaluated once."""
    kind = case["kind"]
    if kind == "boxes":   # the mean of the log-uniform sizes
        lo, hi = case["n_min"], case["n_max"]
        n = case["boxes"] * ((hi - lo) / math.log(hi / lo) if hi > lo else lo)
    else:
        n = case["n"]
    na = n * case.get("fraction", 1.0)
    dens, force = PAIRS_DENSITY * FLOPS_DENSITY, PAIRS_FORCE * FLOPS_FORCE
    if kind in ("step", "boxes"):
        return {"bytes": n * (73 + (12 if case.get("f64") else 0)), "flops": n * (dens + force)}
    if kind == "timebins":
        return {"bytes": n * 73 * 1.111, "flops": n * 1.111 * (dens + force)}
    if kind == "substep":
        return {"bytes": na * 73, "flops": na * (dens + force)}
    if kind == "viscosity":
        return {"bytes": na * 89, "flops": na * (1.5 * dens + 1.05 * force)}
    if kind == "conduction":
        return {"bytes": na * 68, "flops": na * 1.1 * force}
    if kind == "gravity":
        # inside the cutoff sphere of 5.6 spacings, twice that where particles cluster; nodes a quarter
        return {"bytes": n * 16 + na * 20, "flops": na * 1900 * FLOPS_GRAVITY}
    if kind == "adjoint":
        return {"bytes": n * 110, "flops": n * (dens + force + 3 * force)}
    ticks = 1 << case["max_bin"]
    return {"bytes": n * ticks * 80, "flops": n * 1.5 * (dens + force)}


# ---------------------------------------------------------------------------
# 64 bits
# ---------------------------------------------------------------------------

MOST_EXACT = 900_000


def _w(q):
    a, b = (1 - q).clamp_min(0), (0.5 - q).clamp_min(0)
    a2, b2 = a * a, b * b
    return 2 * a2 * a - 8 * b2 * b, 24 * b2 - 6 * a2


def _curve(X):
    """63-bit Morton keys of integer positions in [0, 2^32)."""
    key = torch.zeros(X.shape[0], dtype=torch.int64, device=X.device)
    for b in range(21):
        for a in range(3):
            key |= ((X[:, a] >> (11 + b)) & 1) << (3 * b + 2 - a)
    return key


def _neighbours(x, rows=768):
    """h with (32/3) sum_j w(r_ij/h) = N_t (bisection, then Newton), and the pairs (i, j), j != i, r_ij < h_i, of
    one periodic unit box. Runs of particles along the curve share the candidates around their box."""
    n = x.shape[0]
    order = torch.sort(_curve((x * 2.0 ** 32).long() % (1 << 32))).indices
    h = torch.empty(n, device=x.device, dtype=x.dtype)
    pi, pj = [], []
    for c in range(0, n, rows):
        i = order[c:c + rows]
        lo, hi = x[i].amin(0), x[i].amax(0)
        mid, half = 0.5 * (lo + hi), 0.5 * (hi - lo)
        gap = x - mid
        gap = ((gap - torch.round(gap)).abs() - half).amax(1)   # to the run's box, largest axis
        R = float(torch.quantile(half, 0.5)) * 0.5 + 1e-4
        while True:
            R = min(R, 0.5)
            cand = (gap < R).nonzero()[:, 0]
            r2 = torch.zeros(len(i), len(cand), device=x.device, dtype=x.dtype)
            for a in range(3):
                d = x[cand, a][None, :] - x[i, a][:, None]
                r2 += (d - torch.round(d)) ** 2
            r = r2.sqrt()
            if R >= 0.5 or bool(((32.0 / 3.0) * _w(r / R)[0].sum(1) > N_TARGET).all()):
                break
            R *= 1.6
        lo, hi = r.new_full((len(i), 1), 1e-7).float(), r.new_full((len(i), 1), R).float()
        r32 = r.float()
        for _ in range(24):
            m = 0.5 * (lo + hi)
            small = (32.0 / 3.0) * _w(r32 / m)[0].sum(1, keepdim=True) < N_TARGET
            lo, hi = torch.where(small, m, lo), torch.where(small, hi, m)
        hh = (0.5 * (lo + hi)).double()
        for _ in range(3):   # Newton on the smooth, increasing N(h): quadratic from 1e-6
            w, dw = _w(r / hh)
            N, dN = (32.0 / 3.0) * w.sum(1, keepdim=True), -(32.0 / 3.0) * (r / hh * dw).sum(1, keepdim=True) / hh
            hh = hh - (N - N_TARGET) / dN
        h[i] = hh[:, 0]
        p, q = (r < hh).nonzero(as_tuple=True)
        pi.append(i[p])
        pj.append(cand[q])
    pi, pj = torch.cat(pi), torch.cat(pj)
    keep = pi != pj
    return h, pi[keep], pj[keep]


def _symmetric(pi, pj, n):
    """The pairs with r < max(h_i, h_j), both orders."""
    key = torch.unique(torch.cat([pi * n + pj, pj * n + pi]))
    return key // n, key % n


def _sum(v, i, n):
    return torch.zeros(n, *v.shape[1:], device=v.device, dtype=v.dtype).index_add_(0, i, v)


def _density(x, m, h, pi, pj):
    n = x.shape[0]
    d = x[pj] - x[pi]
    d = d - torch.round(d)
    q = d.norm(dim=1) / h[pi]
    w, dw = _w(q)
    smw = _sum(m[pj] * w, pi, n) + m
    smqdw = _sum(m[pj] * q * dw, pi, n)
    return 8 / math.pi / h ** 3 * smw, -3 * smw / smqdw


def _divcurl(x, m, v, h, rho, pi, pj):
    n = x.shape[0]
    d = x[pj] - x[pi]
    d = d - torch.round(d)
    r = d.norm(dim=1)
    ok = r > 0
    g = torch.where(ok, m[pj] * _w(r / h[pi])[1] / r.clamp_min(1e-300), 0.0)[:, None]
    vij = v[pi] - v[pj]
    c = 8 / math.pi / h ** 4 / rho
    div = _sum((g * vij * -d).sum(1), pi, n)
    curl = _sum(g * torch.linalg.cross(vij, -d), pi, n)
    return -c * div, c * curl.norm(dim=1)


def _force(x, m, v, u, h, rho, omega, pi, pj, alpha=None, divv=None, curlv=None, kappa=None):
    n = x.shape[0]
    P = (GAMMA - 1) * rho * u
    c, A = (GAMMA * P / rho).sqrt(), omega * P / rho ** 2
    d = x[pj] - x[pi]
    d = d - torch.round(d)
    r2 = (d * d).sum(1)
    some = r2 > 0
    r = torch.where(some, r2, 1.0).sqrt()
    F = lambda hh: torch.where(some, 8 / math.pi / hh ** 4 * _w(r / hh)[1] / r, 0.0)
    Fi, Fj = F(h[pi]), F(h[pj])
    vr = -((v[pi] - v[pj]) * d).sum(1)
    w = torch.where(some, vr / r, 0.0)
    vs = c[pi] + c[pj] - 3 * w
    al = 1.0 if alpha is None else 0.5 * (alpha[pi] + alpha[pj])
    Pi = torch.where(w < 0, -al * vs * w / (rho[pi] + rho[pj]), 0.0)
    if divv is not None:
        f = divv.abs() / (divv.abs() + curlv + 1e-4 * c / h)
        Pi = Pi * 0.5 * (f[pi] + f[pj])
    Fb = 0.5 * (Fi + Fj)
    out = {"acc": _sum((m[pj] * (A[pi] * Fi + A[pj] * Fj + Pi * Fb))[:, None] * d, pi, n),
           "dudt": _sum(m[pj] * vr * (A[pi] * Fi + 0.5 * Pi * Fb), pi, n)}
    if vs.requires_grad:
        return out
    out["vsig"] = torch.zeros(n, device=x.device, dtype=x.dtype).scatter_reduce_(0, pi, vs, "amax").clamp_min(0)
    if kappa is not None:
        ks = kappa[pi] + kappa[pj]
        kij = torch.where(ks > 0, 4 * kappa[pi] * kappa[pj] / ks.clamp_min(1e-300), 0.0)
        out["dcond"] = _sum(m[pj] / (rho[pi] * rho[pj]) * kij * (u[pi] - u[pj]) * Fb, pi, n)
    return out


def _exact_step(p):
    x, m, v, u = (p[k].double() for k in ("pos", "mass", "vel", "u"))
    n = x.shape[0]
    h, pi, pj = _neighbours(x)
    rho, omega = _density(x, m, h, pi, pj)
    qi, qj = _symmetric(pi, pj, n)
    return {"h": h, "rho": rho, "omega": omega, **_force(x, m, v, u, h, rho, omega, qi, qj)}


def _exact_viscosity(case, p, gen):
    x, m, v, u = (p[k].double() for k in ("pos", "mass", "vel", "u"))
    n = x.shape[0]
    _randn(gen, n)   # the scatter of the guesses
    alpha = (0.1 + 0.9 * _rand(gen, n)).float().double()
    h, pi, pj = _neighbours(x)
    rho, omega = _density(x, m, h, pi, pj)
    div, curl = _divcurl(x, m, v, h, rho, pi, pj)
    qi, qj = _symmetric(pi, pj, n)
    out = {"h": h, "rho": rho, "omega": omega, "divv": div, "curlv": curl,
           **_force(x, m, v, u, h, rho, omega, qi, qj, alpha, div, curl)}
    c = (GAMMA * (GAMMA - 1) * u).sqrt()
    out["dalpha"] = (-div).clamp_min(0) * (1.0 - alpha) - (alpha - 0.1) * 0.2 * c / h
    return out


def _exact_conduction(case, p, gen):
    x, m, v, u = (p[k].double() for k in ("pos", "mass", "vel", "u"))
    n = x.shape[0]
    _randn(gen, n)   # the scatter of the guesses
    kappa = (10.0 ** (_rand(gen, n) - 1.0)).float().double()
    h, pi, pj = _neighbours(x)
    rho, omega = _density(x, m, h, pi, pj)
    qi, qj = _symmetric(pi, pj, n)
    return _force(x, m, v, u, h, rho, omega, qi, qj, kappa=kappa)


def _exact_adjoint(p, gen):
    x, m, v, u = (p[k].detach().double() for k in ("pos", "mass", "vel", "u"))
    n = x.shape[0]
    ga, gr = (t.double() for t in _seeds(n, gen))
    h0, pi, pj = _neighbours(x)
    qi, qj = _symmetric(pi, pj, n)
    x, m, u = (t.requires_grad_(True) for t in (x, m, u))
    # h as a function of x: one Newton step from the root has the exact first derivative
    d = x[pj] - x[pi]
    d = d - torch.round(d)
    q = d.norm(dim=1) / h0[pi]
    w, dw = _w(q)
    N = (32.0 / 3.0) * (1 + _sum(w, pi, n))
    dN = -(32.0 / 3.0) * _sum((q * dw).detach(), pi, n) / h0
    h = h0 - (N - N.detach()) / dN
    rho, omega = _density(x, m, h, pi, pj)
    out = _force(x, m, v, u, h, rho, omega, qi, qj)
    g = torch.autograd.grad((out["acc"], rho), (x, m, u), (ga, gr))
    return {"acc": out["acc"].detach(), "rho": rho.detach(), "g_pos": g[0], "g_mass": g[1], "g_u": g[2]}


def _tree(pos, m):
    """Quantised positions, Morton order (ties by index) and, per level, node boxes and moments."""
    X = torch.round(pos.double().remainder(1.0) * 2.0 ** 32).long() % (1 << 32)
    order = torch.sort(_curve(X), stable=True).indices
    Xs, ms = X[order], m.double()[order]
    levels = []
    lo = hi = Xs
    mass, com = ms, Xs.double() / 2.0 ** 32
    while True:
        n = lo.shape[0]
        k = -(-n // 8)
        pad = lambda t, v: torch.cat([t, torch.full((k * 8 - n, *t.shape[1:]), v, device=t.device, dtype=t.dtype)])
        com = (pad(mass[:, None] * com, 0).view(k, 8, 3).sum(1)) / pad(mass, 0).view(k, 8).sum(1)[:, None]
        mass = pad(mass, 0).view(k, 8).sum(1)
        lo = pad(lo, (1 << 32) - 1).view(k, 8, 3).amin(1)
        hi = pad(hi, 0).view(k, 8, 3).amax(1)
        levels.append((lo, hi, mass, com))
        if k == 1:
            return order, Xs, ms, levels


def _exact_gravity(case, p):
    order, X, m, levels = _tree(p["pos"], p["mass"])
    n, s = case["n"], _gravity_split(case["n"])
    rci = math.ceil((s["r_cut"] * 2.0 ** 24) ** 2)
    P = round(case["theta"] ** 2 * 65536)
    xs = X.double() / 2.0 ** 32
    act = _first(p, case["fraction"])
    rank = torch.empty_like(order)
    rank[order] = torch.arange(n, device=order.device)
    targets = torch.arange(n, device=order.device) if act is None else rank[act.long()].sort().values
    acc = torch.zeros(n, 3, device=X.device, dtype=torch.float64)
    M32 = (1 << 32) - 1

    def term(t, d, mass):
        r2 = (d * d).sum(1)
        ok = r2 > 0
        r = torch.where(ok, r2, 1.0).sqrt()
        q = (r / s["h_soft"]).clamp_max(1.0)
        Mq = torch.where(q <= 0.5, q ** 3 * (32 / 3 + q * q * (32 * q - 192 / 5)),
                         q ** 3 * (64 / 3 + q * (-48 + q * (192 / 5 - 32 / 3 * q))) - 1 / 15)
        Mq = torch.where(r < s["h_soft"], Mq, torch.ones_like(Mq))
        y = r / (2 * s["r_split"])
        g = torch.special.erfc(y) + 2 / math.sqrt(math.pi) * y * torch.exp(-y * y)
        acc.index_add_(0, order[t], torch.where(ok, mass * Mq * g / r ** 3, 0.0)[:, None] * d)

    for c in range(0, len(targets), 4096):
        t = targets[c:c + 4096]
        node = torch.zeros_like(t)
        for lev in range(len(levels) - 1, -1, -1):   # the root is opened whatever the rule says
            if lev < len(levels) - 1:
                lo, hi, mass, com = levels[lev]
                D2 = torch.zeros_like(t)
                F2, side = torch.zeros_like(t), torch.zeros_like(t)
                for a in range(3):
                    x, l, h = X[t, a], lo[node, a], hi[node, a]
                    out = (x < l) | (x > h)
                    gap = torch.where(out, torch.minimum((l - x) & M32, (x - h) & M32), torch.zeros_like(x))
                    far = torch.where(out, gap + (h - l), torch.maximum(x - l, h - x))
                    D2 += (gap >> 8) ** 2
                    F2 += ((far + 255) >> 8) ** 2
                    side = torch.maximum(side, (h - l) >> 8)
                L2 = side ** 2
                near = D2 < rci
                take = near & (D2 > 0) & (F2 < rci) & (L2 <= D2) if P > 0 else torch.zeros_like(near)
                small = L2.clamp_max(1 << 46) * 65536 <= P * D2.clamp_max(rci)   # (D2 < rci where it counts)
                take = take & small
                d = com[node[take]] - xs[t[take]]
                term(t[take], d - torch.round(d), mass[node[take]])
                go = near & ~take
                t, node = t[go], node[go]
            count = levels[lev - 1][0].shape[0] if lev > 0 else n
            child = node[:, None] * 8 + torch.arange(8, device=node.device)
            ok = child < count
            t = t[:, None].expand(-1, 8)[ok]
            node = child[ok]
        d2 = torch.zeros_like(t)
        for a in range(3):
            d = (X[node, a] - X[t, a]) & M32
            d2 += (torch.minimum(d, (1 << 32) - d) >> 8) ** 2
        ok = (d2 < rci) & (node != t)
        d = xs[node[ok]] - xs[t[ok]]
        term(t[ok], d - torch.round(d), m[node[ok]])
    return {"acc": acc, "n_nodes": None, "n_pairs": None}


def exact(case, seed):
    kind, gen = case["kind"], _gen(seed)
    if kind == "boxes":
        if sum(_box_sizes(case)) > MOST_EXACT:
            return None
        p, offs = _boxes(case, gen)
        parts = [_exact_step({k: v[a:b] for k, v in p.items()}) for a, b in zip(offs, offs[1:])]
        out = {k: torch.cat([q[k] for q in parts]) for k in parts[0]}
    elif kind == "gravity":
        return _exact_gravity(case, _particles(case, gen)) if case["n"] <= 1_600_000 else None
    elif kind in ("kdk", "timebins", "substep") or case.get("fraction", 1.0) != 1.0 or case["n"] > MOST_EXACT:
        return None
    elif kind == "step":
        out = _exact_step(_particles(case, gen))
    elif kind == "viscosity":
        out = _exact_viscosity(case, _particles(case, gen), gen)
    elif kind == "conduction":
        return _exact_conduction(case, _particles(case, gen), gen)
    elif kind == "adjoint":
        return _exact_adjoint(_particles(case, gen), gen)
    else:
        return None
    return {**out, "n_ngb": None, "flags": None}
