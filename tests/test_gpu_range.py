"""Results at the ends of a format's range: boxes, conductivities and densities
whose intermediate values leave the normal numbers or pass any fixed constant,
and sums whose terms cancel to the last bits."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from sph_cases import as_f32, check_force, dev, gpu_density, gpu_force, gpu_grid, host, oracle_all

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    from paper_2003_10850_gb300 import build
    build.build()
    import paper_2003_10850_gb300 as S
    return S


@pytest.fixture(scope="module")
def ctx(S):
    return S.Context(0)


# box 2^54: h about 1.5e15, squared radii above 1e30; box 2^-36: h about 1e-12
@pytest.mark.parametrize("exp", [54, -36])
def test_density_scales_with_the_box(S, ctx, exp):
    """Positions and h times a power of two: every operation of the density pass
    is the same up to that factor (no value leaves the normal range), so h is
    the unit box's times the factor and the counts, sets and Omega are equal,
    to the last bit. 32,768 particles: the member-parallel kernel."""
    f = 2.0 ** exp
    p = as_f32(W.config1(32))
    q = W.Particles(p.pos * f, p.vel, p.mass, p.u, f)
    g1 = gpu_density(S, ctx, gpu_grid(S, ctx, p, S.default_params()), np.full(p.n, 0.08, np.float32),
                     S.default_params())
    params = S.default_params(box=f)
    g2 = gpu_density(S, ctx, gpu_grid(S, ctx, q, params), np.full(p.n, np.float32(0.08) * np.float32(f)), params)
    assert g1["rc"] == 0 and g2["rc"] == 0
    assert np.array_equal(g2["h"].astype(np.float64), g1["h"].astype(np.float64) * f)
    for k in ("n_ngb", "hash", "omega"):
        assert np.array_equal(g1[k], g2[k]), k


@pytest.fixture(scope="module")
def lattice():
    p = as_f32(W.config1(16))
    return p, oracle_all(p)


# masses and densities times 2^-66: rho_i rho_j is subnormal; kappa times 2^-130:
# kappa_i + kappa_j is
@pytest.mark.parametrize("mexp,kexp", [(-66, 0), (0, -130)])
@pytest.mark.parametrize("lists", [True, False])
def test_conduction_with_subnormal_divisors(S, ctx, lattice, mexp, kexp, lists):
    """From the recorded lists and walked, within the force tests' tolerances; a
    conductivity whose products underflow conducts nothing."""
    p, (X, d, _) = lattice
    h, rho, om = (d[k].astype(np.float32) for k in ("h", "rho", "omega"))
    fm, fk = np.float32(2.0 ** mexp), np.float32(2.0 ** kexp)
    kappa = np.random.default_rng(11).uniform(0.1, 2.0, p.n).astype(np.float32) * fk
    q = W.Particles(p.pos, p.vel, p.mass * float(fm), p.u, p.box)
    rq = rho * fm
    f = oracle.force(X, p.vel, q.mass, p.u, h, rq, om)
    co, cs = oracle.conduction(X, q.mass, p.u, h, rq, kappa)
    grid = gpu_grid(S, ctx, q, S.default_params())
    if lists:
        S.density(ctx, grid, dev(h), None, S.default_params(flags=S.SPH_FIXED_H))
    n = p.n
    acc, du, vs = torch.zeros(n, 3, device="cuda"), torch.zeros(n, device="cuda"), torch.zeros(n, device="cuda")
    dc = torch.zeros(n, device="cuda")
    hs = torch.zeros(n, dtype=torch.int64, device="cuda")
    S.sph_hydro_force_conduction(ctx, grid, dev(p.vel), dev(p.u), dev(h), dev(rq), dev(om), None, None, dev(kappa),
                                 None, acc, du, vs, dc, hs, S.default_params())
    rc, st = S.sph_sync_status(ctx, raise_on_error=False)
    assert rc == 0 and (st["list_force"] == n) == lists
    check_force({"acc": host(acc), "dudt": host(du), "vsig": host(vs), "hash": host(hs).view(np.uint64)}, f,
                np.arange(n), 1e-4)
    dcg = host(dc).astype(np.float64)
    if kexp:   # 4 kappa_i kappa_j underflows
        assert np.all(dcg == 0.0)
    else:
        assert np.all(np.abs(dcg - co) <= 1e-4 * cs)


# pairs 3 to 12 integer units apart inside the softening, and 11 to 15 units without
# one: r^3 is subnormal (r below 2.3e-13), the term is not
@pytest.mark.parametrize("soft,units", [(0.01, (3, 5, 8, 12)), (0.0, (11, 12, 13, 15))])
def test_gravity_of_close_pairs_in_a_small_box(S, ctx, soft, units):
    """Counts exact, accelerations within the gravity tests' 2e-5 of the
    per-particle scale."""
    L = 2.0 ** -14
    rng = np.random.default_rng(19)
    n = 512
    pos = np.rint(rng.random((n, 3)) * 2.0 ** 32) * (L * 2.0 ** -32)
    mate = pos[: n // 2].copy()
    mate[:, 0] += np.resize(np.array(units), n // 2) * (L * 2.0 ** -32)
    pos = np.concatenate([pos, mate]) % L
    mass = rng.uniform(0.5, 1.5, len(pos)).astype(np.float32).astype(np.float64) / len(pos)
    sp = dict(theta=0.5, r_split=0.05 * L, r_cut=0.2 * L, h_soft=soft * L)
    o = oracle.gravity(oracle.quantize(pos, L), mass, box=L, **sp)
    grid = S.sph_build_grid(ctx, dev(pos, torch.float64), dev(mass), S.default_params(box=L))
    acc = torch.zeros(len(pos), 3, device="cuda")
    nn, npr = (torch.zeros(len(pos), dtype=torch.int32, device="cuda") for _ in range(2))
    S.sph_gravity(ctx, grid, None, S.gravity_params(**sp), acc, nn, npr)
    S.sph_sync_status(ctx)
    assert np.array_equal(host(nn), o["n_nodes"]) and np.array_equal(host(npr), o["n_pairs"])
    err = np.linalg.norm(host(acc) - o["acc"], axis=1)
    assert np.all(err <= 2e-5 * o["scale"]), (err / o["scale"]).max()


def test_fp64_force_of_mirrored_partners(S, ctx):
    """Fourteen pairs of equal partners on opposite sides of a particle, whose
    terms cancel, and one of mass 2^-40: the sum is its term, which rounding
    the others' sums to 2^-53 of them would bury (their magnitudes are about
    2^40 times it). One term per lane: only the fold over the lanes adds."""
    rng = np.random.default_rng(23)
    o = rng.integers(-60_000, 60_000, (14, 3)) * 2.0 ** -20
    lone = np.array([[31_007, -20_011, 9_001]]) * 2.0 ** -20
    pos = np.concatenate([np.zeros((1, 3)), o, -o, lone]) + 0.5
    n = len(pos)
    mass = np.ones(n)
    mass[-1] = 2.0 ** -40
    h = np.full(n, 0.15, np.float32)
    one = np.ones(n, np.float32)
    p = W.Particles(pos, np.zeros((n, 3)), mass, np.ones(n), 1.0)
    params = S.default_params(flags=S.SPH_FP64)
    g = gpu_force(S, ctx, gpu_grid(S, ctx, p, params), p, h, one, one, params)
    assert g["rc"] == 0
    H, r = float(h[0]), np.linalg.norm(lone[0])
    a, b = max(1 - r / H, 0.0), max(0.5 - r / H, 0.0)
    F = 8 / np.pi * H ** -4 * (24 * b * b - 6 * a * a) / r
    want = mass[-1] * 2 * (params.gamma - 1.0) * F * lone[0]
    assert np.all(np.abs(g["acc"][0] - want) <= 2.0 ** -22 * np.abs(want))
