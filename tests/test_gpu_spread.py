"""Launches with fewer rays than thread slots: every ray once, the same bits
whatever the spread of the rays over warps and SMs."""
import numpy as np
import pytest

import corona_synth as cs
from test_gpu_parity import ctx, rt, tiny  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s_mode", [0, 1, 2])
@pytest.mark.parametrize("nx,ny", [(1, 1), (32, 19), (29, 21), (152, 128), (149, 131), (320, 250)])
def test_spread_of_small_launches(rt, ctx, tiny, nx, ny, s_mode):  # noqa: F811
    """1, 608, 609, 19456, 19519 and 80000 rays: below, at and above one warp
    per scheduler and one wave of thread slots."""
    import torch
    grid = ctx.load(tiny[0])
    v = cs.View(0.3, 0.2, nx, ny, -2.5, 2.5, -2.5, 2.5)
    a = ctx.trace_image(grid, v, [90e6], rt.options(s_mode=s_mode, dtau=2e-2))
    assert ctx.stats()["rays"] == nx * ny
    b = ctx.trace_image(grid, v, [90e6], rt.options(s_mode=s_mode, dtau=2e-2, blocks_per_sm=1, tile=8))
    assert ctx.stats()["rays"] == nx * ny
    torch.cuda.synchronize()
    assert torch.equal(a, b)


@pytest.mark.parametrize("nx,ny", [(1, 1), (32, 19), (29, 21), (90, 70)])
def test_spread_of_the_adjoint(rt, ctx, tiny, nx, ny):  # noqa: F811
    """The gradient of one map is the sum of those of its halves (FP32 atomics
    in any order: 1e-5 of the largest)."""
    import torch
    grid = ctx.load(tiny[0])
    v = cs.View(0.3, 0.2, nx, ny, -2.0, 2.0, -2.0, 2.0)
    w = torch.from_numpy(np.random.default_rng(1).normal(size=(1, ny, nx)).astype(np.float32)).cuda()
    half = (torch.arange(nx * ny, device="cuda").reshape(1, ny, nx) % 2).float()
    _, _, tape = ctx.trace_image_tape(grid, v, [200e6], rt.options(dtau=2e-2, precision=1))
    whole = tape.backward(w)
    parts = [tape.backward(w * half), tape.backward(w * (1 - half))]
    torch.cuda.synchronize()
    tape.free()
    for i in range(2):
        s = parts[0][i] + parts[1][i]
        assert (whole[i] - s).abs().max() <= 1e-5 * whole[i].abs().max()
