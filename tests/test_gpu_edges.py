"""Sizes at which the sort, the active lists, the gravity groups and the double
passes change their route: block and tile edges, remainders, the smallest
sets, lists that overflow."""
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


# one block up to 8,192 keys, then tiles of 4,096: 40,960 and 100,003 make a
# tile look past more than eight predecessors
@pytest.mark.parametrize("n", [1, 31, 255, 257, 4096, 8191, 8192, 8193, 12_289, 40_960, 100_003])
@pytest.mark.parametrize("values", [1, 3, 5000])
def test_sort_sizes(S, n, values):
    """Full-width keys with many repeats: numpy's stable order exactly."""
    rng = np.random.default_rng(n + values)
    keys = rng.integers(0, 2**64, size=values, dtype=np.uint64)[rng.integers(0, values, size=n)]
    order = np.argsort(keys, kind="stable")
    k = torch.from_numpy(keys.view(np.int64)).cuda()
    out, perm = torch.full_like(k, -1), torch.full((n,), -1, dtype=torch.int32, device="cuda")
    S.sph_sort_keys_static(k, out, perm)
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().view(np.uint64), keys[order])
    assert np.array_equal(perm.cpu().numpy(), order.astype(np.int32))


@pytest.mark.parametrize("n", [1, 15, 4095, 4096, 4097, 140_003])
@pytest.mark.parametrize("shift", [0, 3])
def test_active_list_sizes(S, ctx, n, shift):
    """The list of a tick's active particles, its count and its padding, also
    from bins that do not start on a 16-byte boundary."""
    pos = torch.rand(n, 3, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    grid = S.sph_build_grid(ctx, pos, torch.full((n,), 1.0 / n, device="cuda"), S.default_params())
    g = torch.Generator().manual_seed(n)
    bins = torch.randint(0, 5, (n + shift,), dtype=torch.uint8, generator=g).cuda()[shift:]
    act, cnt = torch.full((n,), 7, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    for tick in (0, 1, 6, 8):
        S.sph_active_from_bins(ctx, grid, bins, tick, 3, act, cnt)
        b = host(bins).astype(np.int64).clip(max=3)
        want = np.nonzero(tick % (1 << (3 - b)) == 0)[0]
        got = host(act)
        assert int(cnt.item()) == len(want)
        assert np.array_equal(got[:len(want)], want) and np.all(got[len(want):] == -1)


# all particles in groups of 2 (30,000) or 4 (62,000), then some of them one per warp
@pytest.mark.parametrize("n", [30_000, 62_000])
@pytest.mark.parametrize("theta", [0.0, 0.5, 1.0])
def test_gravity_groups_and_single_walks_agree(S, ctx, n, theta):
    """Node and pair counts are exact whatever the grouping; the accelerations
    differ by the order of FP32 sums of up to some thousand terms with
    compensation per list: 2e-5 of the acceleration scale (the bound of the
    tests against the oracle)."""
    p = as_f32(W.clustered(n, 40, seed=17))
    cell = 1.0 / round(n ** (1 / 3))
    gp = S.gravity_params(G=1.0, theta=theta, r_split=1.25 * cell, r_cut=4.5 * 1.25 * cell, h_soft=2.8 * cell / 30)
    grid = S.sph_build_grid(ctx, dev(p.pos), dev(p.mass), S.default_params())
    res = []
    act = torch.arange(3, n, 7, dtype=torch.int32, device="cuda")
    for a in (None, act):
        acc = torch.zeros(n, 3, device="cuda")
        nn, npair = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
        S.sph_gravity(ctx, grid, a, gp, acc, nn, npair)
        rc, _ = S.sph_sync_status(ctx)
        assert rc == 0
        res.append((acc[act.long()].double(), nn[act.long()], npair[act.long()]))
    assert torch.equal(res[0][1], res[1][1]) and torch.equal(res[0][2], res[1][2])
    a, b = res[0][0], res[1][0]
    scale = a.norm(dim=1) + a.norm(dim=1).median()
    assert float(((a - b).norm(dim=1) / scale).max()) <= 2e-5


def test_fp64_list_overflow(S, ctx):
    """SPH_FP64 with neighbour lists beyond the 128 entries that a warp keeps: at a
    fixed h, sets exact and sums to FP32 output rounding (the bounds of the
    parity tests)."""
    p = as_f32(W.clustered(12_000, 3, seed=9))
    h = np.full(p.n, 0.06, np.float32)
    o = oracle.density(oracle.quantize(p.pos), p.mass, h.astype(np.float64), fixed_h=True)
    params = S.default_params(flags=S.SPH_FP64 | S.SPH_FIXED_H)
    grid = S.sph_build_grid(ctx, dev(p.pos), dev(p.mass), params)
    rho, om = torch.zeros(p.n, device="cuda"), torch.zeros(p.n, device="cuda")
    nn, fl = torch.zeros(p.n, dtype=torch.int32, device="cuda"), torch.zeros(p.n, dtype=torch.uint8, device="cuda")
    hs = torch.zeros(p.n, dtype=torch.int64, device="cuda")
    S.sph_density(ctx, grid, dev(h), None, rho, om, nn, fl, hs, params)
    S.sph_sync_status(ctx)
    assert o["n_ngb"].max() > 1000
    assert np.array_equal(host(nn), o["n_ngb"])
    assert np.array_equal(host(hs).view(np.uint64), o["hash"])
    assert np.abs(host(rho) / o["rho"] - 1).max() <= 2e-7
    some = o["n_ngb"] > 0   # alone within h, Omega has no value (1 + h/(3 rho) d rho/dh = 0)
    assert np.abs(host(om) / o["omega"] - 1)[some].max() <= 1e-6
