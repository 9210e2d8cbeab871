"""The batched launch, whose cones go through their phases independently: more
cones than a warp looks at once, cones of one bundle and one particle beside
large ones, step counts from 1 up (cones finish at different times), repeated
and smaller batches on the same context, against each cone's own trace.  Both
sum the same FP32 terms, split differently: 1e-7 of a bundle's differential
deflection, a tenth of mu - 1 < 1, so 1e-6 of mu leaves a margin."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


def cones(count, seed):
    g = inputs.rng(inputs.BASE_SEED + seed)
    out = []
    for i in range(count):
        n = int(g.choice([1, 7, 256, 700, 5000]))
        nb = int(g.choice([1, 2, 33, 128, 129, 300]))
        pos = inputs.quantize(np.array([0.0, 0.0, 700.0]) + 0.5 * g.normal(size=(n, 3)))
        out.append(dict(pos=pos, mass=1e11 / n, soft=0.3, theta=4e-4 * g.normal(size=(nb, 2)),
                        z_s=float(g.uniform(0.3, 0.9)), n_steps=int(g.choice([1, 2, 5, 12]))))
    return out


@pytest.mark.parametrize("n_ring", [4, 8, 5])
@pytest.mark.parametrize("count", [1, 31, 70])
def test_independent_cones(n_ring, count):
    import paper_1110_4894_gb300 as P
    cs = cones(count, count)
    ctx = P.Context(0)
    ctx.set_cosmology(0.3, 0.7, 0.7)
    for i, c in enumerate(cs):
        ctx.load_particles(i, c["pos"], c["mass"], c["soft"])
    kw = dict(n_ring=n_ring, theta_r=5e-6)
    batch = [dict(field_id=i, z_s=c["z_s"], theta=c["theta"], n_steps=c["n_steps"]) for i, c in enumerate(cs)]
    one = [ctx.trace(i, c["z_s"], c["theta"], n_steps=c["n_steps"], want_rays=True, **kw) for i, c in enumerate(cs)]
    for part in (batch, batch[: max(1, count // 3)], batch):
        for got, ref in zip(ctx.trace_batch(part, want_rays=True, **kw), one):
            assert np.array_equal(got["flags"], ref["flags"]) and np.array_equal(got["steps"], ref["steps"])
            assert np.max(np.abs(got["mu"] / ref["mu"] - 1)) < 1e-6
    ctx.close()


def test_repeated_batches_are_the_same_bits():
    """the order in which blocks take items changes no sum"""
    import paper_1110_4894_gb300 as P
    cs = cones(40, 9)
    ctx = P.Context(0)
    ctx.set_cosmology(0.3, 0.7, 0.7)
    for i, c in enumerate(cs):
        ctx.load_particles(i, c["pos"], c["mass"], c["soft"])
    batch = [dict(field_id=i, z_s=c["z_s"], theta=c["theta"], n_steps=c["n_steps"]) for i, c in enumerate(cs)]
    first = ctx.trace_batch(batch, n_ring=4, theta_r=5e-6)
    for _ in range(4):
        for a, b in zip(ctx.trace_batch(batch, n_ring=4, theta_r=5e-6), first):
            assert all(np.array_equal(a[k], b[k]) for k in a)
    ctx.close()
