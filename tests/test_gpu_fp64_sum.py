"""The all-FP64 pair sum where its particle loop and splits end: field sizes
around the unroll of 4, the tile of 128 and one wave of splits, against the
oracle's compensated sums.  Each of n terms carries about 6 roundings and the
sum n / 2, of terms of one order of magnitude: n * 1.2e-16 + 1e-15 bounds it,
relative to the sum of the terms' magnitudes."""
import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 4, 5, 127, 128, 129, 131, 3041, 20000])
@pytest.mark.parametrize("points", [1, 255, 257])
@pytest.mark.parametrize("varied", [False, True])
def test_fp64_sum_edges(n, points, varied):
    import paper_1110_4894_gb300 as P
    g = inputs.rng(inputs.BASE_SEED + n)
    pos = inputs.quantize(np.array([0.0, 0.0, 800.0]) + 0.3 * g.normal(size=(n, 3)))
    mass = 1e10 * (g.uniform(0.5, 2.0, n) if varied else np.ones(n))
    soft = g.uniform(0.002, 0.02, n) if varied else 0.01
    pts = inputs.quantize(np.array([0.0, 0.0, 800.0]) + 0.5 * g.normal(size=(points, 3)))
    ctx = P.Context(0, precision=P.FP64)
    ctx.load_particles(0, pos, mass, soft)
    got = ctx.potential(0, pts)
    ctx.close()
    ref = oracle.potential(oracle.MassField(pos, mass, soft), pts)
    d = pos[None] - pts[:, None]
    inv = ((d * d).sum(-1) + np.broadcast_to(soft, (n,)) ** 2) ** -0.5
    scale = oracle.mu_G() * np.stack([(mass * inv).sum(1)] + [(mass * inv ** 3 * np.abs(d[..., k])).sum(1) for k in range(3)], 1)
    assert np.max(np.abs(got - ref) / scale) <= 1.2e-16 * n + 1e-15


def test_fp64_particle_on_the_point_is_infinite():
    """no softening and no distance: an infinite potential, as before a NaN gradient"""
    import paper_1110_4894_gb300 as P
    ctx = P.Context(0, precision=P.FP64)
    ctx.load_particles(0, np.array([[0.0, 0.0, 8.0]]), np.array([1e10]), 0.0)
    out = ctx.potential(0, np.array([[0.0, 0.0, 8.0], [0.0, 1.0, 8.0]]))
    ctx.close()
    assert out[0, 0] == -np.inf and np.isnan(out[0, 1:]).all() and np.isfinite(out[1]).all()
