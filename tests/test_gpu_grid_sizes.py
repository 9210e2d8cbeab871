"""Grids of any size, against the sum over a few particles that sit on nodes: a
particle on a node gives all its mass to it, and a point on a node reads that
node, so the grid's field is the Plummer sum itself, whatever the path of the
build (spectra of two kernels kept and turned up to 406 nodes a side, each
kernel's own transforms beyond; FFTs of more than 2^31 elements from 813 on).
The node table of a mixed context is FP32: 6e-8 of a value, and as much again
for each of the weights of its interpolation; 1e-6 of the sum's terms leaves a
margin."""
import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [37, 406, 408, 819])
def test_particles_on_nodes(n):
    import torch

    import paper_1110_4894_gb300 as P
    # FFT buffers, values, table, and the work areas of the plans
    if torch.cuda.mem_get_info()[0] < 440 * n ** 3:
        pytest.skip("needs %.0f GB of device memory" % (440e-9 * n ** 3))
    h = 0.0625
    g = inputs.rng(inputs.BASE_SEED + n)
    k = np.concatenate([g.integers(0, n, (5, 3)), [[0, n - 1, n // 3]]])
    at = np.concatenate([g.integers(0, n, (400, 3)), [[0, 0, 0], [n - 1, 0, 0], [0, n - 1, 0], [n - 1, n - 1, n - 1]]])
    lo, mass, soft = np.array([-8.0, 16.0, 512.0]), 1e12 * g.uniform(0.5, 2.0, len(k)), 4 * h
    ctx = P.Context(0)
    ctx.set_cosmology(0.3, 0.7, 0.7)
    ctx.load_grid(0, lo + h * k, mass, soft, lo, h, n)
    got = ctx.potential(0, lo + h * at)
    ctx.close()
    d = h * (at[:, None] - k[None]).astype(float)
    w = oracle.mu_G() * mass / np.sqrt((d ** 2).sum(-1) + soft ** 2)
    w3 = w[..., None] * d / ((d ** 2).sum(-1) + soft ** 2)[..., None]
    assert np.all(np.abs(got[:, 0] + w.sum(1)) <= 1e-6 * w.sum(1))
    assert np.all(np.abs(got[:, 1:] - w3.sum(1)) <= 1e-6 * np.linalg.norm(w3, axis=-1).sum(1)[:, None])
