"""Calls on a GPU with little memory left: what a grid build keeps only for speed
must not take the room of what it cannot do without."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


def leave(free):
    """takes all but free bytes of the GPU's memory"""
    import torch
    torch.cuda.empty_cache()
    return torch.empty(max(0, torch.cuda.mem_get_info()[0] - int(free)), dtype=torch.uint8, device="cuda")


def release():
    import torch
    torch.cuda.empty_cache()


def test_grid_build_without_room_for_the_spectra():
    """the kernel spectra (128 bytes a node) are left out where they do not fit beside FFT buffers, values, table
    and particles: the build works, through the kernels' own transforms, whose node values are the same but for
    the rounding of FFTs (2^-53 times their 30 levels, of the largest value: 1e-11 leaves a margin)"""
    import paper_1110_4894_gb300 as P
    n, h, npart = 192, 0.0625, 1 << 24
    g = inputs.rng(inputs.BASE_SEED + 81)
    some = g.uniform(0.0, (n - 1) * h, (4096, 3))
    pos, mass = np.tile(some, (npart // 4096, 1)), np.full(npart, 1e7)
    at = g.uniform(0.0, (n - 1) * h, (2000, 3))
    needed = n ** 3 * (8 + 64 + 2 * 64 * (n + 1) / n + 32 + 32 + 64) + 32 * npart
    spectra = 128 * n * n * (n + 1)
    res = []
    for tight in (False, True):
        ctx = P.Context(0, precision=P.FP64)
        ctx.set_cosmology(0.3, 0.7, 0.7)
        filler = leave(needed + 0.45 * spectra) if tight else None
        ctx.load_grid(0, pos, mass, 0.05, [0.0, 0.0, 0.0], h, n)
        del filler
        release()
        res.append(ctx.potential(0, at))
        ctx.close()
    assert np.max(np.abs(res[0])) > 0.0
    assert np.all(np.abs(res[1] - res[0]) <= 1e-11 * np.max(np.abs(res[0]), axis=0))


@pytest.mark.parametrize("bad", [None, "pos", "mass", "soft", "box"])
def test_load_beside_a_field_that_leaves_no_room(bad):
    """a new field whose upload does not fit beside the old one: valid particles take its place, invalid ones are
    found on the host before it goes.  The old one holds 16 bytes or more a particle, an upload takes 32 to 40"""
    import paper_1110_4894_gb300 as P
    n = 1 << 22
    g = inputs.rng(inputs.BASE_SEED + 82)
    L = inputs.box_length(8.0)
    pos, mass, soft = g.random((n, 3)) * L * 0.999, g.uniform(1e8, 2e8, n), g.uniform(0.01, 0.02, n)
    old = np.tile(pos, (4, 1))
    vol = dict(replicated=True, box_length=L, rot=np.eye(3, dtype=np.int32)[None], shift=np.zeros((1, 3)))
    at = g.random((50, 3))
    ctx = P.Context(0)
    ctx.load_particles(0, pos, mass, soft, **vol)
    want = ctx.potential(0, at)
    ctx.load_particles(0, old, 1e8, 0.02)
    before = ctx.potential(0, at)
    if bad == "pos":
        pos[n // 2, 1] = np.inf
    elif bad == "mass":
        mass[n - 1] = -1.0
    elif bad == "soft":
        soft[n // 3] = np.nan
    elif bad == "box":
        pos[n - 1, 2] = 1.5 * L
    filler = leave(20 * n)
    if bad is None:
        ctx.load_particles(0, pos, mass, soft, **vol)
        assert np.array_equal(ctx.potential(0, at), want)
    else:
        message = {"pos": "non-finite", "mass": "masses must", "soft": "softening", "box": "outside [0, L]"}[bad]
        with pytest.raises(P.Rt3dError) as e:
            ctx.load_particles(0, pos, mass, soft, **vol)
        assert message in str(e.value)
        assert np.array_equal(ctx.potential(0, at), before)
    del filler
    release()
    ctx.close()
