"""FP64 traces through at most 64 particles run in one launch (k_few_trace):
against the same trace stage by stage (kernel timing asks for that) and against
the oracle.  Both sum the same FP64 terms, the ray's offset rounded once more or
less: positions differ by rounding of 1e-13 Mpc over separations of 5e-3 Mpc
and more, 1e-10 of mu at the most."""
import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu


# 65 particles: past the limit, both are the kernels of a stage; bundles around
# the six (rings of 4) or three (rings of 8) of a warp
@pytest.mark.parametrize("n", [1, 2, 31, 64, 65])
@pytest.mark.parametrize("n_ring,bundles", [(3, 1), (4, 6), (4, 7), (5, 11), (8, 3), (8, 4)])
@pytest.mark.parametrize("varied", [False, True])
def test_few_particles(cosmo, n, n_ring, bundles, varied):
    import paper_1110_4894_gb300 as P
    g = inputs.rng(inputs.BASE_SEED + n)
    pos = inputs.quantize(np.array([0.0, 0.0, 1000.0]) + 0.3 * g.normal(size=(n, 3)))
    mass = 1e13 / n * (g.uniform(0.5, 2.0, n) if varied else np.ones(n))
    soft = g.uniform(0.02, 0.05, n) if varied else 0.03
    theta = 3e-4 * g.normal(size=(bundles, 2))
    kw = dict(n_ring=n_ring, theta_r=5e-6, schedule=1, n_steps=60, lens_chi=1000.0, asinh_s=0.05)
    res = []
    for timed in (0, 1):
        ctx = P.Context(0, precision=P.FP64, time_kernels=timed)
        ctx.set_cosmology(0.3, 0.7, 0.7)
        ctx.load_particles(0, pos, mass, soft)
        res.append(ctx.trace(0, 0.5, theta, want_rays=True, **kw))
        res[-1]["interactions"] = ctx.stats()["interactions"]
        ctx.close()
    a, b = res
    assert np.array_equal(a["flags"], b["flags"]) and np.array_equal(a["steps"], b["steps"])
    assert a["interactions"] == b["interactions"]
    o = oracle.trace(cosmo, oracle.MassField(pos, mass, soft), 0.5, theta, **kw)
    for other in (b["mu"], o.mu):
        assert np.max(np.abs(a["mu"] / other - 1)) < 1e-10


def test_few_particles_in_pieces(cosmo):
    """advanced 7 stages at a time (through step boundaries) as in one go"""
    import torch

    import paper_1110_4894_gb300 as P
    pos = inputs.quantize(np.array([[0.0, 0.0, 1000.0], [0.2, 0.1, 700.0]]))
    theta = torch.tensor([[3e-4, 0.0], [0.0, -2e-4], [1e-4, 1e-4]], dtype=torch.float64, device="cuda")
    kw = dict(n_ring=4, theta_r=5e-6, n_steps=20)
    out = [torch.empty((3, 6), dtype=torch.float64, device="cuda") for _ in range(2)]
    ctx = P.Context(0, precision=P.FP64)
    ctx.set_cosmology(0.3, 0.7, 0.7)
    ctx.load_particles(0, pos, 1e13, 0.03)
    ctx.trace_device(0, 0, 0.5, 3, theta.data_ptr(), out[0].data_ptr(), **kw)
    ctx.trace_begin(0, 0, 0.5, 3, theta.data_ptr(), **kw)
    for _ in range(5):
        ctx.trace_advance(0, 7)
    ctx.trace_end(0, out[1].data_ptr())
    torch.cuda.synchronize()
    ctx.close()
    assert torch.equal(out[0], out[1])


# one launch up to 22 particles, and up to 64 from 64 rays an SM on (9728 on GB300's 152)
@pytest.mark.parametrize("n,bundles,one", [(22, 3, True), (23, 3, False), (23, 1945, False), (23, 1946, True),
                                           (64, 1945, False), (64, 1946, True), (65, 1946, False)])
def test_where_one_launch_takes_over(n, bundles, one):
    import torch

    import paper_1110_4894_gb300 as P
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    bundles = bundles * sms // 152 + (bundles == 1946 and sms != 152)
    g = inputs.rng(inputs.BASE_SEED + n)
    pos = inputs.quantize(np.array([0.0, 0.0, 1000.0]) + 0.3 * g.normal(size=(n, 3)))
    theta = 3e-4 * g.normal(size=(bundles, 2))
    kw = dict(n_ring=4, theta_r=5e-6, schedule=1, n_steps=60, lens_chi=1000.0, asinh_s=0.05)
    res = []
    for timed in (0, 1):
        ctx = P.Context(0, precision=P.FP64, time_kernels=timed)
        ctx.set_cosmology(0.3, 0.7, 0.7)
        ctx.load_particles(0, pos, 1e13 / n, 0.03)
        res.append(ctx.trace(0, 0.5, theta, **kw))
        assert (ctx.stats()["threads_per_block"] == 32) == (one and not timed)
        ctx.close()
    # (of 1 / mu, the Jacobian's determinant, as some of these many bundles may lie near a critical line)
    a, b = 1 / res[0]["mu"], 1 / res[1]["mu"]
    assert np.all(np.abs(a - b) <= 1e-10 * (1 + np.abs(b)))
