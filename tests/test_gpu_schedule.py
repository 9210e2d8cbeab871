"""The step table and the redshifts behind it, summed by groups of lanes
(rt3d_schedule), against the oracle's quadrature."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# fewer and more blocks than steps, one to ninety panels per redshift, the
# first panel alone (z_s = 0.01) and integrals longer than one round of lanes.
# Boole's rule with 4 panels a step leaves 6 (h / l)^6 for quadrature intervals
# h = chi_s / 16 n and a^2 varying over l ~ c / H(z) / 3: below 1e-9 for each
# of these; a distance is one rounding of a 25-term FP64 sum, below 1e-13.
@pytest.mark.parametrize("z_s,n", [(0.01, 1), (0.16, 3), (0.5, 24), (0.5, 333), (1.8, 150), (0.5, 5003)])
@pytest.mark.parametrize("kind", [0, 1])
def test_step_table_matches_oracle(cosmo, z_s, n, kind):
    import paper_1110_4894_gb300 as P
    if kind == 1 and n < 100:
        pytest.skip("asinh steps this long are not resolved by the rule")
    ctx = P.Context(0)
    ctx.set_cosmology(0.3, 0.7, 0.7)
    chi_s = cosmo.chi(z_s)
    dl, chi = ctx.schedule(z_s, kind, n, 0.5 * chi_s, 0.2 * chi_s)
    ref, _ = cosmo.schedule(chi_s, kind, n, 0.5 * chi_s, 0.2 * chi_s)
    ctx.close()
    assert abs(chi / chi_s - 1) < 1e-13
    assert np.max(np.abs(dl / ref - 1)) < 1e-9
