"""Mid-size traces through a mean-subtracted box: the kernels of a stage (pair
sum, prism, integrator stage) take little longer for 1024 bundles than for 256,
as neither fills the GPU.  Where blocks of the next kernels were let in beside the
running ones, the larger trace took 3.5 times the smaller one's time (20.5 against
5.8 ms; 6.0 against 5.6 without)."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


def test_kernels_of_a_stage_do_not_crowd_each_other():
    import paper_1110_4894_gb300 as P
    L = inputs.box_length(100.0)
    g = inputs.rng(inputs.BASE_SEED + 91)
    pos = np.minimum(inputs.quantize(g.random((500, 3)) * L), L - inputs.QUANTUM)
    rot, shift = inputs.replicas(49, L, 14)
    ctx = P.Context(0)
    ctx.set_cosmology(0.3, 0.7, 0.7)
    ctx.load_particles(0, pos, 1e10, 0.03, replicated=True, box_length=L, rot=rot, shift=shift, mean_subtract=True)
    best = []
    for bundles in (256, 1024):
        theta = 3e-4 * g.normal(size=(bundles, 2))
        times = []
        for _ in range(6):
            ctx.trace(0, 0.5, theta, n_ring=8, theta_r=5e-6, n_steps=30)
            times.append(ctx.stats()["device_ms"])
        best.append(min(times))
    ctx.close()
    assert best[1] < 2.0 * best[0]
