"""Traces with few bundles, whose pair sum puts one ray on a lane
(k_force_bundle1): its operations, their order and the anchors are those of
the two-bundle kernel, which an explicit split count asks for, so with one tile
per split both give the same bits, and both meet the oracle at the gates of the
mixed path."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


def case(n, varied, box):
    g = inputs.rng(inputs.BASE_SEED + n)
    if box:
        L = inputs.box_length(40.0)
        pos = np.minimum(inputs.quantize(g.random((n, 3)) * L), L - inputs.QUANTUM)
        rot, shift = inputs.replicas(49, L, 5)
        vol = dict(replicated=True, box_length=L, rot=rot, shift=shift, mean_subtract=True)
    else:
        pos, vol = inputs.quantize(np.array([0.0, 0.0, 1000.0]) + 0.5 * g.normal(size=(n, 3))), {}
    mass = 3e10 * (g.uniform(0.5, 2.0, n) if varied else np.ones(n))
    soft = g.uniform(0.01, 0.03, n) if varied else 0.02
    return pos, mass, soft, vol


# bundles: one, a warp's worth (6 of 5 rays, 3 of 9) and one more, a block's (25, 14) and one more, more than
# the 128 bundles that share an anchor; particles: below, at and above whole tiles of 256
@pytest.mark.parametrize("n_ring,bundles", [(4, 1), (4, 6), (4, 7), (4, 25), (4, 26), (4, 131), (8, 3), (8, 4), (8, 15),
                                            (8, 129)])
@pytest.mark.parametrize("n", [3, 256, 517])
@pytest.mark.parametrize("varied", [False, True])
@pytest.mark.parametrize("box", [False, True])
def test_one_ray_lanes_give_the_same_bits(n_ring, bundles, n, varied, box):
    import paper_1110_4894_gb300 as P
    pos, mass, soft, vol = case(n, varied, box)
    theta = np.array([3e-4, -2e-4]) + 2e-4 * inputs.rng(7).normal(size=(bundles, 2))
    res = []
    for opt in (dict(), dict(splits=(n + 255) // 256)):
        ctx = P.Context(0, **opt)
        ctx.set_cosmology(0.3, 0.7, 0.7)
        ctx.load_particles(0, pos, mass, soft, **vol)
        res.append(ctx.trace(0, 0.5, theta, want_rays=True, n_ring=n_ring, theta_r=5e-6, n_steps=12))
        assert ctx.stats()["splits"] == (n + 255) // 256
        ctx.close()
    for k in res[0]:
        assert np.array_equal(res[0][k], res[1][k]), k


def test_statistics_name_the_block_that_ran():
    """one-ray lanes run in blocks of one warp (bundles that fit it) or four, two-bundle threads in blocks of 64, and
    the traces whose rays evaluate the field themselves in blocks of one warp"""
    import paper_1110_4894_gb300 as P
    pos, mass, soft, vol = case(517, False, False)
    shapes = {}
    for name, opt, bundles in (("warp", {}, 6), ("block", {}, 7), ("threads", dict(splits=3), 7),
                               ("few", dict(precision=P.FP64), 7), ("grid", {}, 7)):
        ctx = P.Context(0, **opt)
        ctx.set_cosmology(0.3, 0.7, 0.7)
        if name == "grid":
            ctx.load_grid(0, pos, mass, soft, [-2.0, -2.0, 998.0], 4.0 / 15, 16)
        else:
            ctx.load_particles(0, pos[:3] if name == "few" else pos, mass[:3] if name == "few" else mass, soft, **vol)
        ctx.trace(0, 0.5, 2e-4 * inputs.rng(7).normal(size=(bundles, 2)), n_ring=4, theta_r=5e-6, n_steps=3)
        st = ctx.stats()
        ctx.close()
        shapes[name] = (st["rays_per_thread"], st["threads_per_block"], st["splits"])
    assert shapes == {"warp": (5, 32, 3), "block": (5, 128, 3), "threads": (5, 64, 3), "few": (1, 32, 1),
                      "grid": (1, 32, 1)}


@pytest.mark.parametrize("box", [False, True])
def test_captured_trace_replays(box):
    """the overlapped launches of a trace, captured into a CUDA graph and replayed, give the same bits"""
    import torch

    import paper_1110_4894_gb300 as P
    pos, mass, soft, vol = case(700, False, box)
    theta = torch.from_numpy(np.array([3e-4, -2e-4]) + 2e-4 * inputs.rng(7).normal(size=(5, 2))).cuda()
    out = [torch.zeros((5, 6), dtype=torch.float64, device="cuda") for _ in range(2)]
    ctx = P.Context(0)
    ctx.set_cosmology(0.3, 0.7, 0.7)
    ctx.load_particles(0, pos, mass, soft, **vol)

    def trace(o):
        ctx.trace_device(torch.cuda.current_stream().cuda_stream, 0, 0.5, 5, theta.data_ptr(), o.data_ptr(), n_ring=4,
                         theta_r=5e-6, n_steps=12)

    trace(out[0])  # sizes the context's scratch
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        trace(out[1])
    for _ in range(3):
        out[1].zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out[0], out[1])
    ctx.close()
