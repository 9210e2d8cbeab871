"""The muPDF kernel at the edges of its chunks, of its shared-memory bins and of
its FP32 bin estimate, against the oracle: whole numbers equal, moments to
rounding (a sum of n FP64 terms of one sign: n / 2 ulp at most)."""
import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu


def values(n, seed, lo, hi, bins):
    """magnifications with every kind of entry: 1e-3 to 1e-12 off the bin edges
    (the two sides' log10 agree to 1e-15), both parities, zeros, infinities,
    NaN, far out of range"""
    g = inputs.rng(seed)
    mu = 10.0 ** g.normal(0.0, 0.1, n)
    edge = 10.0 ** (np.log10(lo) + (np.log10(hi) - np.log10(lo)) / bins * g.integers(0, bins + 1, n))
    k = g.integers(0, 12, n)
    mu = np.where(k < 3, edge * (1.0 + g.choice((-1, 1), n) * 10.0 ** g.uniform(-12, -3, n)), mu)
    mu = np.where(k == 3, -mu, mu)
    odd = np.array([0.0, np.inf, -np.inf, np.nan, 1e-35, 1e35, 1e-200, 3.0])
    mu = np.where(g.random(n) < 0.02, odd[g.integers(0, odd.size, n)], mu)
    return mu, np.where(g.random(n) < 0.01, g.integers(0, 8, n), 0).astype(np.int32)


@pytest.mark.parametrize("n", [0, 1, 1023, 1024, 1025, 300001, 1024 * 1024 + 77])
@pytest.mark.parametrize("bins,lo,hi", [(1, 0.5, 5.0), (200, 0.5, 5.0), (1024, 0.9, 1.1), (1025, 0.9, 1.1),
                                        (100000, 0.5, 5.0)])
def test_mupdf_edges(n, bins, lo, hi):
    import paper_1110_4894_gb300 as P
    mu, flags = values(n, inputs.BASE_SEED + n + bins, lo, hi, bins)
    ctx = P.Context(0)
    c, w, s = ctx.histogram(mu, flags, bins, lo, hi)
    ctx.close()
    co, wo, so = oracle.histogram(mu, flags, bins, lo, hi)
    assert np.array_equal(c, co) and np.array_equal(w, wo)
    for k in ("n_used", "n_under", "n_over", "n_neg", "n_bad"):
        assert s[k] == so[k], k
    tol = 1.2e-16 * max(n, 8)
    for k in ("W_total", "mean_w", "sigma_w"):
        assert s[k] == so[k] or abs(s[k] / so[k] - 1) <= tol, k
