"""The replica transform in 32-bit arithmetic, over every signed permutation,
with shifts and positions at the edges of their ranges and points far outside
the box (whose offsets need 64 bits), against the oracle's FP64 placement: the
grid holds these positions exactly, so the FP64 potential agrees to the
rounding of a sum of n terms."""
import itertools

import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [8.0, 142.5, 500.0])
def test_every_signed_permutation(L):
    import paper_1110_4894_gb300 as P
    L = inputs.box_length(L)
    rots = []
    for perm in itertools.permutations(range(3)):
        for sign in itertools.product((1, -1), repeat=3):
            R = np.zeros((3, 3), np.int32)
            R[np.arange(3), perm] = sign
            rots.append(R)
    rot = np.array(rots)
    n_rep, q = len(rot), inputs.QUANTUM
    g = inputs.rng(inputs.BASE_SEED + 48)
    shift = inputs.quantize(g.random((n_rep, 3)) * (L - q))
    shift[::3] = 0.0
    shift[1::3] = L - q
    edge = np.array([0.0, q, 0.5 * L, 0.5 * L + q, L - q])
    pos = np.concatenate([edge[g.integers(0, 5, (60, 3))], inputs.quantize(g.random((200, 3)) * (L - q))])
    mass = g.uniform(0.5, 2.0, len(pos)) * 1e12
    rep = np.repeat(np.arange(n_rep, dtype=np.int32), 3)
    pts = np.stack([g.uniform(-0.5, 0.5, rep.size) * L, g.uniform(-0.5, 0.5, rep.size) * L,
                    (rep + g.random(rep.size)) * L], 1)
    pts[::3] += 3.0 * L * g.choice((-1, 1), (n_rep, 3))  # outside the replica
    ctx = P.Context(0, precision=P.FP64)
    soft = 0.05 * L
    ctx.load_particles(0, pos, mass, soft, replicated=True, box_length=L, rot=rot, shift=shift)
    got = ctx.potential(0, pts, rep)
    ctx.close()
    ref = oracle.potential(oracle.MassField(pos, mass, soft, replicated=True, L=L, rot=rot, shift=shift), pts, rep)
    for k in range(4):
        assert np.max(np.abs(got[:, k] - ref[:, k])) < 1e-12 * np.max(np.abs(ref[:, k]))
