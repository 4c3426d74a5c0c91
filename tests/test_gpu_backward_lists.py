"""The adjoint from the recorded neighbour lists (sph_backward after an
all-active density call) against the walk (the same call on a grid built
without lists), and against a state the lists were not made for.

Both sum the same FP32 pair terms with compensation; they differ in the
rounding of the separations (2^-24 of the leaf size in the walk) and of the
sums. Tolerance: that of the adjoint tests against the FP64 reference, the
99th percentile <= 5e-5 and the maximum <= 3e-3 of |ref| + median, twice (each
side is allowed that much).
"""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from sph_cases import as_f32, dev, host

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


def _grads(S, ctx, grid, p, h, d, params, seed=3):
    g = torch.Generator().manual_seed(seed)
    abar, rbar = torch.randn(p.n, 3, generator=g).cuda(), torch.randn(p.n, generator=g).cuda()
    out = [torch.empty(p.n, 3, device="cuda"), torch.empty(p.n, device="cuda"), torch.empty(p.n, device="cuda")]
    S.sph_backward(ctx, grid, dev(p.vel), dev(p.u), h, d["rho"], d["omega"], abar, rbar, *out, params)
    rc, _ = S.sph_sync_status(ctx)
    assert rc == 0
    return [host(t).astype(np.float64) for t in out]


def _check(a, b):
    for x, y in zip(a, b):
        e = (np.abs(x - y) / (np.abs(y) + np.median(np.abs(y)))).reshape(len(y), -1).max(1)
        assert np.quantile(e, 0.99) <= 1e-4 and e.max() <= 6e-3, (np.quantile(e, 0.99), e.max())


# 2,051: a last octet and warp partly filled; 4,097 and 20,000 clustered: extra
# partners, and particles whose list is longer than 128
@pytest.mark.parametrize("n,blobs", [(2051, 6), (4097, 8), (20_000, 30)])
def test_lists_and_walk_agree(S, ctx, n, blobs):
    p = as_f32(W.clustered(n, blobs, seed=71))
    res = []
    for flags in (0, S.SPH_NO_LISTS):
        params = S.default_params(flags=flags)
        grid = S.sph_build_grid(ctx, dev(p.pos), dev(p.mass), params)
        h = torch.zeros(p.n, device="cuda")
        d = S.density(ctx, grid, h, None, params)
        res.append(_grads(S, ctx, grid, p, h, d, params))
    _check(*res)


def test_lists_of_another_state_are_not_used(S, ctx):
    """h changed after the density call: the lists must not serve, and the
    result is bit for bit the walk's on a grid without lists."""
    p = as_f32(W.clustered(4097, 8, seed=72))
    res = []
    for flags in (0, S.SPH_NO_LISTS):
        params = S.default_params(flags=flags)
        grid = S.sph_build_grid(ctx, dev(p.pos), dev(p.mass), params)
        h = torch.zeros(p.n, device="cuda")
        d = S.density(ctx, grid, h, None, params)
        h[17] *= 1.01
        if flags == 0:
            keep = (h.clone(), {k: v.clone() for k, v in d.items()})
        res.append(_grads(S, ctx, grid, p, keep[0], keep[1], params))
    for a, b in zip(*res):
        assert np.array_equal(a, b)


def _served(a, b):
    """Where dL/du differs from the walk's: its sums are the particle's own pairs
    only, so a particle that walks has the walk's bits, and one served from the
    lists (exact separations, another order) mostly not."""
    return a[1] != b[1]


def _both(S, ctx, p, params, density, build=None):
    """Gradients on a grid with lists and on one without, at the state that the
    density calls on the first leave."""
    build = build or (lambda params: S.sph_build_grid(ctx, dev(p.pos), dev(p.mass), params))
    grid, walk = build(params), build(S.default_params(flags=S.SPH_NO_LISTS))
    h = torch.zeros(p.n, device="cuda")
    d = density(grid, h)
    return [_grads(S, ctx, g, p, h, d, params) for g in (grid, walk)], host(h)


def test_particles_whose_lists_overflow_walk(S, ctx):
    """A clump of 64 in a sparse shell whose h reaches it: the clump has more than
    128 extra partners and walks in all three passes, the rest reads its lists."""
    rng = np.random.default_rng(12)
    c = np.full(3, 0.5)
    v = rng.standard_normal((160, 3))
    shell = c + v / np.linalg.norm(v, axis=1)[:, None] * rng.uniform(0.05, 0.15, (160, 1))
    bg = rng.uniform(0, 1, (20000, 3))
    pos = np.concatenate([c + 0.001 * rng.standard_normal((64, 3)), shell, bg[np.linalg.norm(bg - c, axis=1) > 0.3]])
    n = len(pos)
    p = as_f32(W.Particles(pos, rng.normal(0, 0.1, (n, 3)), np.full(n, 1.0 / n), rng.uniform(0.5, 1.5, n), 1.0))
    params = S.default_params()
    (a, b), h = _both(S, ctx, p, params, lambda g, h: S.density(ctx, g, h, None, params))
    oi, oj = oracle.pair_list(oracle.quantize(p.pos), h.astype(np.float64))
    r = np.linalg.norm((p.pos[oi] - p.pos[oj] + 0.5) % 1.0 - 0.5, axis=1)
    far = (r >= h[oi] * 1.00001) & (r < h[oj] * 0.99999)
    over = np.bincount(oi[far], minlength=n) > 128
    assert over[:64].sum() > 16
    served = _served(a, b)
    assert not served[over].any() and served[64:].mean() > 0.5, (served[over].sum(), served[64:].mean())
    _check(a, b)


def test_lists_in_two_boxes(S, ctx):
    boxes = [as_f32(W.clustered(n, 5, seed=75 + n)) for n in (3001, 6000)]
    p = W.Particles(*(np.concatenate([getattr(b, k) for b in boxes]) for k in ("pos", "vel", "mass", "u")), 1.0)
    params = S.default_params()
    build = lambda q: S.sph_build_grid_batched(ctx, dev(p.pos), dev(p.mass), [0, 3001, 9001], [1.0, 1.0], q)
    (a, b), _ = _both(S, ctx, p, params, lambda g, h: S.density(ctx, g, h, None, params), build)
    assert _served(a, b).mean() > 0.5
    _check(a, b)


def test_lists_of_a_partial_call(S, ctx):
    """After SPH_PARTIAL_LISTS on the densest fifth: those particles read their
    lists, every other one walks."""
    p = as_f32(W.clustered(50_000, 40, seed=73))
    params = S.default_params()
    sel = {}

    def density(grid, h):
        d = S.density(ctx, grid, h, None, params)
        if "act" not in sel:
            hh = host(h)
            sel["act"] = np.nonzero(hh <= np.quantile(hh, 0.2))[0].astype(np.int32)
        part = S.default_params(flags=S.SPH_FIXED_H | S.SPH_PARTIAL_LISTS)
        S.density(ctx, grid, h, dev(sel["act"], torch.int32), part)
        return d

    (a, b), _ = _both(S, ctx, p, params, density)
    on = np.zeros(p.n, bool)
    on[sel["act"]] = True
    served = _served(a, b)
    assert not served[~on].any() and served[on].mean() > 0.5, (served[~on].sum(), served[on].mean())
    _check(a, b)
