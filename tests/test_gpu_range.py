"""Results at the ends of the FP32 range: boxes, conductivities and densities
whose intermediate values leave the normal numbers or pass any fixed constant."""
import numpy as np
import pytest

import workloads as W
from sph_cases import as_f32, gpu_density, gpu_grid

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
