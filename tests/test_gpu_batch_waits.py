"""The waits of the batched launch.  An idle block waits for an event at most as
long as the watchdog allows, and an expired one ends the whole launch at the items in
hand."""
import time

import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


def context(P, **opt):
    ctx = P.Context(0, **opt)
    ctx.set_cosmology(0.3, 0.7, 0.7)
    g = inputs.rng(inputs.BASE_SEED + 61)
    ctx.load_particles(0, inputs.quantize(np.array([0.0, 0.0, 700.0]) + 0.5 * g.normal(size=(2000, 3))), 5e7, 0.3)
    return ctx


def test_expired_watchdog_ends_the_launch():
    """one cone of two items at most: all other blocks are idle from the start, and the first of them to run out
    of a limit of one microsecond ends a launch that takes seconds otherwise"""
    import paper_1110_4894_gb300 as P
    theta = 4e-4 * inputs.rng(2).normal(size=(128, 2))
    kw = dict(n_ring=4, theta_r=5e-6)
    long, short = ([dict(field_id=0, z_s=0.5, theta=theta, n_steps=n)] for n in (20000, 12))
    ctx, limited = context(P), context(P, watchdog_s=1e-6)
    ref = ctx.trace_batch(short, **kw)[0]
    t0 = time.perf_counter()
    ctx.trace_batch(long, **kw)
    whole = time.perf_counter() - t0
    for _ in range(2):  # the context stays usable, and expires again
        t0 = time.perf_counter()
        with pytest.raises(P.Rt3dError) as e:
            limited.trace_batch(long, **kw)
        cut = time.perf_counter() - t0
        assert e.value.code == P._binding.ETIMEOUT
        assert cut < 0.25 * whole
    one = limited.trace(0, 0.5, theta, n_steps=12, **kw)
    assert np.max(np.abs(one["mu"] / ref["mu"] - 1)) < 1e-6
    limited.close()
    for k, v in ctx.trace_batch(short, **kw)[0].items():
        assert np.array_equal(v, ref[k]), k
    ctx.close()


@pytest.mark.parametrize("cones", [1, 2, 33])
def test_no_block_sleeps_through_a_phase(cones):
    """cones of one force item and one stage item: each phase is opened by the block that ran the one before, and
    whoever finds no work has to wake when it opens.  4000 phases a cone under a limit that one missed wake-up of
    the last waiting block would exceed."""
    import paper_1110_4894_gb300 as P
    theta = 4e-4 * inputs.rng(3).normal(size=(5, 2))
    kw = dict(n_ring=4, theta_r=5e-6)
    batch = [dict(field_id=0, z_s=0.5, theta=theta, n_steps=500)] * cones
    ctx = context(P, watchdog_s=0.5)
    ctx.load_particles(0, inputs.quantize(np.array([[0.0, 0.0, 700.0], [0.1, 0.2, 700.5]])), 5e7, 0.3)
    runs = [ctx.trace_batch(batch, **kw) for _ in range(3)]
    one = ctx.trace(0, 0.5, theta, n_steps=500, **kw)
    ctx.close()
    for run in runs:
        for out in run:
            assert np.array_equal(out["mu"], runs[0][0]["mu"])
    assert np.max(np.abs(runs[0][0]["mu"] / one["mu"] - 1)) < 1e-6
