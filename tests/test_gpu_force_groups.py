"""The force walked in groups (k_force_mp) against the oracle: sets large enough
for it (8 x 48 active particles per SM, the size taken from the device), in
every variant of the pair term, from a grid without lists and for an active
subset of a larger grid; and lists padded to their capacity with a count one
below and one at the device-side rule.

Tolerances: those of the force tests (1e-4 of the per-particle pair-term
scale, pair sets exact).
"""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from sph_cases import as_f32, check_force, dev, gpu_force, gpu_grid, host

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


@pytest.fixture(scope="module")
def least():
    return 8 * 48 * torch.cuda.get_device_properties(0).multi_processor_count


@pytest.fixture(scope="module")
def state(least):
    p = as_f32(W.clustered(2 * least + 3001, 60, seed=207))
    X = oracle.quantize(p.pos)
    d = oracle.density(X, p.mass, None, tol=1e-6)
    h, rho, om = (d[k].astype(np.float32) for k in ("h", "rho", "omega"))
    dv, cv = oracle.divcurl(X, p.vel, p.mass, h, rho)
    rng = np.random.default_rng(17)
    return dict(p=p, X=X, h=h, rho=rho, om=om, dv=dv.astype(np.float32), cv=cv.astype(np.float32),
                alpha=rng.uniform(0.02, 1.5, p.n).astype(np.float32), kappa=rng.uniform(0.1, 2.0, p.n).astype(np.float32))


@pytest.fixture(scope="module")
def grid(S, ctx, state):
    return gpu_grid(S, ctx, state["p"], S.default_params(flags=S.SPH_NO_LISTS))


def _force(S, ctx, grid, s, variant, switch, act, want_hash):
    p, n = s["p"], s["p"].n
    acc, du, vs = torch.zeros(n, 3, device="cuda"), torch.zeros(n, device="cuda"), torch.zeros(n, device="cuda")
    dc = torch.zeros(n, device="cuda")
    hs = torch.zeros(n, dtype=torch.int64, device="cuda") if want_hash else None
    a = None if act is None else dev(act, torch.int32)
    base = [ctx, grid, dev(p.vel), dev(p.u), dev(s["h"]), dev(s["rho"]), dev(s["om"])]
    sw = [dev(s["dv"]), dev(s["cv"])] if switch else [None, None]
    params = S.default_params()
    if variant == "conduction":
        S.sph_hydro_force_conduction(*base, *sw, dev(s["kappa"]), a, acc, du, vs, dc, hs, params)
    elif variant == "alpha":
        S.sph_hydro_force_visc(*base, dev(s["alpha"]), *sw, a, acc, du, vs, hs, params)
    elif switch:
        S.sph_hydro_force_balsara(*base, *sw, a, acc, du, vs, hs, params)
    else:
        S.sph_hydro_force(*base, a, acc, du, vs, hs, params)
    rc, st = S.sph_sync_status(ctx, raise_on_error=False)
    assert rc == 0 and st["list_force"] == 0
    g = {"acc": host(acc), "dudt": host(du), "vsig": host(vs)}
    if want_hash:
        g["hash"] = host(hs).view(np.uint64)
    return g, host(dc).astype(np.float64), st


@pytest.mark.parametrize("switch", [False, True])
@pytest.mark.parametrize("variant", ["scalar", "alpha", "conduction"])
def test_groups_in_every_variant(S, ctx, state, grid, least, variant, switch):
    """All particles, and a random half of them with the rest inactive."""
    s, p = state, state["p"]
    sw = {"divv": s["dv"], "curlv": s["cv"]} if switch else {}
    if variant == "alpha":
        sw["alpha"] = s["alpha"].astype(np.float64)
    f = oracle.force(s["X"], p.vel, p.mass, p.u, s["h"], s["rho"], s["om"], **sw)
    half = W.sample_indices(p.n, least + 1500, seed=5).astype(np.int32)
    for act in (None, half):
        idx = np.arange(p.n) if act is None else act
        for want_hash in (True, False):
            g, dc, st = _force(S, ctx, grid, s, variant, switch, act, want_hash)
            check_force(g, f, idx, 1e-4, check_hash=want_hash)
            assert st["force_pairs"] == int(f["n_pairs"][idx].sum())
            if variant == "conduction":
                co, cs = oracle.conduction(s["X"], p.mass, p.u, s["h"], s["rho"], s["kappa"])
                assert np.all(np.abs(dc - co)[idx] <= 1e-4 * cs[idx] + 1e-30)


@pytest.mark.parametrize("span", [8, 512, 4096])
def test_groups_of_other_spans(S, ctx, state, grid, least, span):
    """Groups confined to aligned runs of 8, 512 or 4096 sorted particles."""
    s, p = state, state["p"]
    f = oracle.force(s["X"], p.vel, p.mass, p.u, s["h"], s["rho"], s["om"])
    half = W.sample_indices(p.n, least + 1500, seed=6).astype(np.int32)
    g = gpu_force(S, ctx, grid, p, s["h"], s["rho"], s["om"], S.default_params(group_size=span), active=half)
    assert g["rc"] == 0
    check_force(g, f, half, 1e-4)


def test_padded_lists_on_both_sides_of_the_rule(S, ctx, state, grid, least):
    """The host sees only the capacity (every particle); the device's count
    decides. A group tests its candidates for all of its members, the
    one-particle walk only each particle's own, so the tests per particle tell
    which kernel ran."""
    s, p = state, state["p"]
    f = oracle.force(s["X"], p.vel, p.mass, p.u, s["h"], s["rho"], s["om"])
    order = np.argsort(p.pos[:, 0], kind="stable").astype(np.int32)   # a slab: full groups
    tests = {}
    for count in (least - 1, least):
        act = np.sort(order[:count])
        pad = np.concatenate([act, np.full(p.n - count, -1, np.int32)])
        g = gpu_force(S, ctx, grid, p, s["h"], s["rho"], s["om"], S.default_params(), active=pad)
        assert g["rc"] == 0
        check_force(g, f, act, 1e-4)
        assert g["stats"]["force_pairs"] == int(f["n_pairs"][act].sum())
        tests[count] = g["stats"]["pair_tests"] / count
    print("pair tests per particle", tests)
    assert tests[least] > 1.1 * tests[least - 1], tests
