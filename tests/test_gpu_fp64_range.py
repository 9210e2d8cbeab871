"""1 / r of the FP64 pair sum over the range of FP64 numbers: one particle at the
origin and points along an axis, so that the separation is exact.  r^2 is rounded
once (2^-54 of 1 / r), the correction of the hardware's estimate once (2^-53), the
product with the mass and the mass itself once each: less than 4 x 2^-53 of the
potential.  Below 2^-511 r^2 is subnormal, a multiple of 2^-1074, and the
potential as uncertain as that makes it; beyond 2^512 it is infinite and the
potential and its gradient vanish."""
import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu


def potential(r):
    """at distances r; every 256th point, the anchor of its block's offsets, is the origin itself"""
    import paper_1110_4894_gb300 as P
    at = np.arange(len(r)) + np.arange(len(r)) // 255 + 1
    pts = np.zeros((at[-1] + 1, 3))
    pts[at, at % 3] = r
    ctx = P.Context(0, precision=P.FP64)
    ctx.load_particles(0, np.zeros((1, 3)), np.array([1e12]), 0.0)
    out = ctx.potential(0, pts)
    ctx.close()
    return out[at]


def error(r, phi):
    """relative error of phi against the quotient in extended arithmetic"""
    from fractions import Fraction
    m = Fraction(oracle.mu_G() * 1e12)
    return np.array([abs(float(Fraction(p) * Fraction(x) / -m - 1)) for x, p in zip(r.tolist(), phi.tolist())])


def test_inverse_distance_over_all_decades():
    g = inputs.rng(inputs.BASE_SEED + 71)
    s = np.where(g.random(6000) < 0.5, -1.0, 1.0)
    far, near = 2.0 ** g.uniform(-510, 510, 3000), 10.0 ** g.uniform(-6, 4, 3000)
    r = s * np.concatenate([far, near])
    assert error(np.abs(r), potential(r)[:, 0]).max() <= 4 * 2.0 ** -53


def test_inverse_distance_at_the_ends_of_the_range():
    r = np.array([1.3e154, 1.2e154, 1.0e154, 7.0e153, 5e153, 2.0 ** 511])
    assert error(r, potential(r)[:, 0]).max() <= 4 * 2.0 ** -53
    r = np.array([1.4e-154, 1e-155, 3e-157, 1e-160])
    assert np.all(error(r, potential(r)[:, 0]) <= 2.0 ** -1074 / (r * r) + 4 * 2.0 ** -53)


def test_no_pull_from_an_infinite_square_distance():
    r = np.array([1.4e154, 1e155, -1e200, 1e250, -1e290])
    assert np.all(potential(r) == 0.0)
