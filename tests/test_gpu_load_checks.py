"""rt3d_load_particles checks its inputs on the device: the first invalid
particle decides the message, as a loop over them would; a refused load leaves
the slot's field as it was; sizes around the blocks and chains of the scan."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture
def ctx():
    import paper_1110_4894_gb300 as P
    c = P.Context(0)
    yield c
    c.close()


def particles(n):
    g = inputs.rng(inputs.BASE_SEED + n)
    return inputs.quantize(g.random((n, 3)) * 8.0), g.uniform(1e10, 2e10, n), g.uniform(0.01, 0.02, n)


@pytest.mark.parametrize("n", [2, 255, 1024, 1025, 200000])
@pytest.mark.parametrize("what,message", [("pos", "non-finite particle position"), ("mass", "masses must be > 0"),
                                          ("soft", "softening must be >= 0"), ("box", "outside [0, L]")])
def test_refused_loads(ctx, n, what, message):
    import paper_1110_4894_gb300 as P
    pos, mass, soft = particles(n)
    ctx.load_particles(0, pos, mass, soft)
    at = np.array([[4.0, 5.0, 6.0]])
    before = ctx.potential(0, at)
    i = n - 1 if n < 1000 else n // 2
    vol = {}
    if what == "pos":
        pos[i, 2] = np.nan
        mass[min(i + 1, n - 1)] = -1.0  # a later particle's, or the same one's, later check
    elif what == "mass":
        mass[i] = 0.0
        soft[i] = -1.0
    elif what == "soft":
        soft[i] = np.inf
    else:
        pos[i, 1] = 8.5
        vol = dict(replicated=True, box_length=8.0, rot=np.eye(3, dtype=np.int32)[None], shift=np.zeros((1, 3)))
    with pytest.raises(P.Rt3dError) as e:
        ctx.load_particles(0, pos, mass, soft, **vol)
    assert message in str(e.value)
    assert np.array_equal(ctx.potential(0, at), before)


@pytest.mark.parametrize("n", [1, 31, 1023, 1024, 1025, 155649])
def test_scan_of_a_field(ctx, n):
    """extent and total mass: the field of a mean-subtracted box is that of its particles minus a prism with the
    box's mean density (sums of n FP64 terms: n * 1.2e-16), found again from two boxes that differ in it alone"""
    pos, mass, soft = particles(n)
    L = inputs.box_length(8.0)
    vol = dict(replicated=True, box_length=L, rot=np.eye(3, dtype=np.int32)[None], shift=np.zeros((1, 3)))
    at = np.array([[0.5, 0.25, 3.0]])
    import paper_1110_4894_gb300 as P
    c = P.Context(0, precision=P.FP64)
    c.load_particles(0, pos, mass, 0.02, mean_subtract=True, **vol)
    c.load_particles(1, pos, mass, 0.02, mean_subtract=False, **vol)
    import oracle
    prism = oracle.prism(np.array([-L / 2, -L / 2, 0.0]), np.array([L / 2, L / 2, L]), at[0])
    got = (c.potential(0, at) - c.potential(1, at))[0]
    c.close()
    want = oracle.mu_G() * mass.sum() / L ** 3 * np.asarray(prism)
    assert np.max(np.abs(got - want)) <= (1e-12 + 2.4e-16 * n) * np.max(np.abs(want))
