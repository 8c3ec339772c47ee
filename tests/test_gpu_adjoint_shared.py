"""The adjoint of retraced steps, whose neighbours the lanes of a warp share:
warps that hold one ray, warps full of rays where single lanes ask, where
several passes are needed, and where every lane takes its own neighbours."""
import numpy as np
import pytest

import corona_synth as cs
from test_gpu_curvature import corona
from test_gpu_parity import ctx, rt  # noqa: F401

pytestmark = pytest.mark.gpu


def gradient(rt, ctx, grid, v, freqs, w, opts):  # noqa: F811
    import torch
    _, _, tape = ctx.trace_image_tape(grid, v, freqs, rt.options(precision=1, **opts))
    out = tape.backward(w)
    torch.cuda.synchronize()
    tape.free()
    return [x.cpu().numpy().astype(np.float64) for x in out]


@pytest.mark.parametrize("lat", [0.2, 1.45, np.pi / 2])
def test_neighbours_of_one_ray(rt, ctx, orc, lat):  # noqa: F811
    """112 rays, one to a warp, every step retraced, on cells that hold hundreds
    of steps: the neighbours' parts are 1 / eps times what is left of a pair, so
    a pair must cancel before it meets other sums.  Against the oracle's tape
    adjoint; bar 1e-5 relative L2: FP32's 6e-8 a term over the square root of the
    3e4 terms that a node sums."""
    opts = dict(dtau=1.2e-2)
    g = corona(5, 3, 4)
    v = cs.View(0.4, lat, 8, 7, -1.7, 1.87, -1.53, 1.7)
    freqs = [60e6, 300e6]
    w = np.random.default_rng(3).normal(size=(2, v.ny, v.nx))
    got = gradient(rt, ctx, ctx.load(g), v, freqs, w, opts)
    ref = orc.backward(orc.grid_field(g), v, freqs, w.reshape(2, -1), orc.default_options(tau_stop=30.0, **opts))[:2]
    rel = [np.linalg.norm(a - b) / np.linalg.norm(b) for a, b in zip(got, ref)]
    print(lat, "relative L2", rel)
    assert max(rel) <= 1e-5, rel


@pytest.mark.parametrize("shape,nx,ny,opts", [
    ((24, 16, 32), 160, 128, dict(dtau=1.6e-2)),           # every lane asks at every step: four passes
    ((96, 64, 128), 160, 128, dict(dtau=4e-3)),            # none to many lanes ask, one pass and more
    ((24, 16, 32), 256, 256, dict(dtau=1.6e-2)),           # blocks of 512 threads
    ((24, 16, 32), 256, 256, dict(dtau=1.6e-2, s_mode=2)),
])
def test_full_warps(rt, ctx, shape, nx, ny, opts):  # noqa: F811
    """The gradient of a dense view is the sum of those of its blocks of 512
    pixels, whose launches have one ray to a warp.  The pixels are 2^-6 R_sun,
    so that a block's rays are the view's bit for bit; what differs is the order
    of FP32 sums: 6e-8 over the square root of 1e5 terms of a node, 2e-5."""
    grid = ctx.load(corona(*shape))
    d = 2.0 ** -6
    x0, y0 = -nx // 2 * d + d, -ny // 2 * d - 3 * d
    view = lambda ix, iy, n, m: cs.View(0.3, 0.25, n, m, x0 + ix * d, x0 + (ix + n) * d, y0 + iy * d, y0 + (iy + m) * d)
    w = np.random.default_rng(11).normal(size=(1, ny, nx))
    whole = gradient(rt, ctx, grid, view(0, 0, nx, ny), [90e6], w, opts)
    parts = [0.0, 0.0]
    for iy in range(0, ny, 16):
        for ix in range(0, nx, 32):
            p = gradient(rt, ctx, grid, view(ix, iy, 32, 16), [90e6], w[:, iy:iy + 16, ix:ix + 32], opts)
            parts = [a + b for a, b in zip(parts, p)]
    rel = [np.linalg.norm(a - b) / np.linalg.norm(b) for a, b in zip(whole, parts)]
    print(shape, opts, "relative L2", rel)
    assert max(rel) <= 2e-5, rel


@pytest.mark.parametrize("opts", [dict(dtau=4e-3), dict(dtau=8e-3, s_mode=2)])
def test_few_weights(rt, ctx, opts):  # noqa: F811
    """Three weighted rays in a view of 20480: most warps of their blocks have
    nothing to do at any step.  Against the single rays (as test_full_warps)."""
    grid = ctx.load(corona(24, 16, 32))
    d = 2.0 ** -6
    pix = [(3, 5, 1.0), (80, 64, -2.0), (159, 127, 0.5)]
    w = np.zeros((1, 128, 160))
    parts = [0.0, 0.0]
    for ix, iy, c in pix:
        w[0, iy, ix] = c
        v = cs.View(0.3, 0.25, 1, 1, -1.25 + ix * d, -1.25 + (ix + 1) * d, -1.0 + iy * d, -1.0 + (iy + 1) * d)
        parts = [a + b for a, b in zip(parts, gradient(rt, ctx, grid, v, [90e6], np.full((1, 1, 1), c), opts))]
    whole = gradient(rt, ctx, grid, cs.View(0.3, 0.25, 160, 128, -1.25, 1.25, -1.0, 1.0), [90e6], w, opts)
    for a, b in zip(whole, parts):
        assert np.linalg.norm(a - b) <= 2e-5 * np.linalg.norm(b)
