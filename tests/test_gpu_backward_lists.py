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
