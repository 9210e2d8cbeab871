"""The integrator stage's sum of split partials around its groups of 16 and 64
rows: the same trace with any number of splits.  The partials are compensated
pairs (FP32 pair sums) or FP64 sums, so regrouping moves the field by 2^-45 or
less, except the potential, an FP32 sum per split (1e-6 of itself, which enters
the geodesics at 1e-11 of the path): mu stays within 1e-9 of its largest
value, on this weak field."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("bundles", [1, 7, 40])
def test_any_number_of_splits(precision, bundles):
    import paper_1110_4894_gb300 as P
    n = 256 * 130
    g = inputs.rng(inputs.BASE_SEED + 130)
    pos = inputs.quantize(np.array([0.0, 0.0, 1000.0]) + 0.5 * g.normal(size=(n, 3)))
    theta = np.array([3e-4, -2e-4]) + 2e-4 * g.normal(size=(bundles, 2))
    res = []
    for splits in (8, 9, 15, 16, 17, 63, 64, 65, 128, 130):
        ctx = P.Context(0, precision=P.FP64 if precision == "fp64" else P.MIXED, splits=splits)
        ctx.set_cosmology(0.3, 0.7, 0.7)
        ctx.load_particles(0, pos, 1e9, 0.05)
        res.append(ctx.trace(0, 0.5, theta, n_ring=4, theta_r=5e-6, n_steps=6)["mu"])
        ctx.close()
    for r in res[1:]:
        assert np.max(np.abs(r - res[0])) <= 1e-9 * np.max(np.abs(res[0]))


# (40 bundles give no SM two of the stage's blocks of 32 rays, 1100 do: 96 and 64
# rows in flight)
@pytest.mark.parametrize("bundles", [40, 1100])
def test_splits_around_the_rows_in_flight(bundles):
    import paper_1110_4894_gb300 as P
    n = 256 * 130
    g = inputs.rng(inputs.BASE_SEED + 131)
    pos = inputs.quantize(np.array([0.0, 0.0, 1000.0]) + 0.5 * g.normal(size=(n, 3)))
    theta = np.array([3e-4, -2e-4]) + 2e-4 * g.normal(size=(bundles, 2))
    res = []
    for splits in (9, 63, 64, 65, 95, 96, 97, 130):
        ctx = P.Context(0, precision=P.MIXED, splits=splits)
        ctx.set_cosmology(0.3, 0.7, 0.7)
        ctx.load_particles(0, pos, 1e9, 0.05)
        res.append(ctx.trace(0, 0.5, theta, n_ring=4, theta_r=5e-6, n_steps=6)["mu"])
        ctx.close()
    for r in res[1:]:
        assert np.max(np.abs(r - res[0])) <= 1e-9 * np.max(np.abs(res[0]))


# (from 256 splits on, and up to 4864 / 4 rays, a kernel of its own adds the
# partials up, in tiles of 48 rows and blocks of 16 rays)
@pytest.mark.parametrize("bundles,n_ring", [(1, 4), (3, 4), (16, 8), (33, 4), (130, 8), (243, 4)])
@pytest.mark.parametrize("splits", [256, 287, 288, 289, 480, 700])
def test_many_splits(bundles, n_ring, splits):
    import paper_1110_4894_gb300 as P
    n = 256 * splits - 3
    g = inputs.rng(inputs.BASE_SEED + 132)
    pos = inputs.quantize(np.array([0.0, 0.0, 1000.0]) + 0.5 * g.normal(size=(n, 3)))
    theta = np.array([3e-4, -2e-4]) + 2e-4 * g.normal(size=(bundles, 2))
    res = []
    for s in (64, splits):
        ctx = P.Context(0, precision=P.MIXED, splits=s)
        ctx.set_cosmology(0.3, 0.7, 0.7)
        ctx.load_particles(0, pos, 1e9 * 33280 / n, 0.05)
        res.append(ctx.trace(0, 0.5, theta, n_ring=n_ring, theta_r=5e-6, n_steps=6)["mu"])
        ctx.close()
    assert np.max(np.abs(res[1] - res[0])) <= 1e-9 * np.max(np.abs(res[0]))


# (96 rows in flight: from 256 splits on, where the partials are not added up
# beforehand, which is above 4864 / 4 rays or in FP64, and up to 152 blocks of 32 rays)
@pytest.mark.parametrize("precision,bundles", [("mixed", 256), ("mixed", 900), ("fp64", 1), ("fp64", 40), ("fp64", 900)])
@pytest.mark.parametrize("splits", [256, 287, 288, 289, 480])
def test_many_splits_in_the_stage(precision, bundles, splits):
    import paper_1110_4894_gb300 as P
    per = 256 if precision == "mixed" else 64
    n = per * splits - 3
    g = inputs.rng(inputs.BASE_SEED + 133)
    pos = inputs.quantize(np.array([0.0, 0.0, 1000.0]) + 0.5 * g.normal(size=(n, 3)))
    theta = np.array([3e-4, -2e-4]) + 2e-4 * g.normal(size=(bundles, 2))
    res = []
    for s in (64, splits):
        ctx = P.Context(0, precision=P.FP64 if precision == "fp64" else P.MIXED, splits=s)
        ctx.set_cosmology(0.3, 0.7, 0.7)
        ctx.load_particles(0, pos, 1e9 * 33280 / n, 0.05)
        res.append(ctx.trace(0, 0.5, theta, n_ring=4, theta_r=5e-6, n_steps=6)["mu"])
        used = ctx.stats()["splits"]
        ctx.close()
    assert used == splits
    assert np.max(np.abs(res[1] - res[0])) <= 1e-9 * np.max(np.abs(res[0]))
