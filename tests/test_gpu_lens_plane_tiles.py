"""The lens-plane pair sum stages only a tile's particles on the plane: fields
whose tiles hold none, one, all or some of them, in any order, against the
oracle (the mixed path's gates: 1e-5 of the deflection's rms, 1e-4 of mu)."""
import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ring", [4, 8])
@pytest.mark.parametrize("layout", ["sorted", "reversed", "mixed", "one_far"])
@pytest.mark.parametrize("n", [1, 63, 256, 1025])
@pytest.mark.parametrize("slices", [1, 4])
def test_planes_of_partly_filled_tiles(cosmo, n_ring, layout, n, slices):
    import paper_1110_4894_gb300 as P
    g = inputs.rng(inputs.BASE_SEED + n)
    z = g.uniform(400.0, 1600.0, n)
    if layout == "sorted":  # whole tiles on one plane
        z = np.sort(z)
    elif layout == "reversed":
        z = np.sort(z)[::-1]
    elif layout == "one_far":  # planes with a single particle
        z = np.full(n, 500.0)
        z[n // 2] = 1500.0
    pos = inputs.quantize(np.stack([0.5 * g.normal(size=n), 0.5 * g.normal(size=n), z], 1))
    mass, soft = g.uniform(0.5, 2.0, n) * 1e12 / max(n, 16), 0.05
    theta = 2e-4 * g.normal(size=(9, 2))
    kw = dict(n_ring=n_ring, theta_r=5e-6, slices=slices)
    ctx = P.Context(0)
    ctx.set_cosmology(0.3, 0.7, 0.7)
    ctx.load_particles(0, pos, mass, soft)
    r = ctx.multiplane(0, 0.5, theta, **kw)
    ctx.close()
    o = oracle.multiplane(cosmo, oracle.MassField(pos, mass, soft), 0.5, theta, **kw)
    assert np.max(np.abs(r["mu"] / o.mu - 1)) < 1e-4
    assert np.max(np.abs(r["kappa"] - o.kappa)) < 1e-4
