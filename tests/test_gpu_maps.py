"""Beam convolution and disk mean at the edges of their kernels' tiles and
windows, against the definitions of the oracle package."""
import numpy as np
import pytest

import corona_synth as cs
from test_gpu_parity import ctx, rt  # noqa: F401

pytestmark = pytest.mark.gpu


def maps(nf, ny, nx, seed=0):
    rng = np.random.default_rng(seed)
    return (1e6 * (rng.random((nf, ny, nx)) - 0.1)).astype(np.float32)


@pytest.mark.parametrize("nx,ny,baseline", [
    (1, 1, 15e3), (127, 9, 15e3), (128, 8, 15e3), (129, 33, 5e3), (33, 129, 1e3), (300, 40, 300.0), (40, 300, 300.0)])
def test_beam_tiles_and_windows(rt, ctx, nx, ny, baseline):  # noqa: F811
    """Windows of one to many times 64 taps, ragged tiles.  Bar: the float32
    result and scratch (2 x 6e-8), expf and the normalisation (2 x 1e-7)."""
    import torch

    from oracle import beam_convolve
    e = 0.01
    v = cs.View(0.0, 0.0, nx, ny, -e * nx, e * nx, -e * ny, e * ny)
    f = [40e6, 200e6, 800e6]
    tb = maps(3, ny, nx)
    out = ctx.beam_convolve(v, torch.from_numpy(tb).cuda(), f, baseline)
    ref = beam_convolve(v, tb.astype(np.float64), f, baseline).reshape(tb.shape)
    assert np.abs(out.cpu().numpy() - ref).max() <= 4e-7 * np.abs(tb).max()


def test_beam_non_finite(rt, ctx):  # noqa: F811
    """An infinite or NaN pixel spoils the outputs that its beam reaches, and
    no others; values whose weighted sum passes FP32's range stay finite."""
    import torch
    v = cs.View(0.0, 0.0, 200, 70, -2.0, 2.0, -0.7, 0.7)
    tb = torch.full((1, 70, 200), 3e38, device="cuda")
    assert torch.isfinite(ctx.beam_convolve(v, tb, [60e6], 5e3)).all()
    tb = torch.from_numpy(maps(1, 70, 200)).cuda()
    base = ctx.beam_convolve(v, tb, [200e6], 15e3)
    for bad in (float("inf"), float("nan")):
        t = tb.clone()
        t[0, 30, 100] = bad
        out = ctx.beam_convolve(v, t, [200e6], 15e3)
        spoiled = ~torch.isfinite(out)
        assert spoiled[0, 30, 100] and spoiled.sum() < 400
        assert (torch.isinf(out) if bad == float("inf") else torch.isnan(out))[spoiled].all()
        assert torch.equal(out[~spoiled], base[~spoiled])


@pytest.mark.parametrize("nx,ny,extent,off,radius", [
    (1, 1, 1.0, 0.0, 0.5), (64, 64, 2.5, 0.0, 0.5), (97, 61, 3.0, 0.0, 1.5), (512, 300, 3.0, 0.0, 0.5),
    (50, 50, 3.0, 0.0, 100.0), (50, 50, 3.0, 0.0, 1e-3), (64, 48, 0.5, 5.0, 4.9), (64, 48, -1.0, 0.3, 0.7)])
def test_disk_mean_boxes(rt, ctx, nx, ny, extent, off, radius):  # noqa: F811
    """Disks that fill, leave or miss the image, flipped axes and an off-centre
    view.  Bar: the FP64 sum's own rounding."""
    import torch

    from oracle import disk_mean_tb
    v = cs.View(0.0, 0.0, nx, ny, off - extent, off + extent, -extent, extent)
    tb = maps(3, ny, nx, 1)
    out = ctx.disk_mean_tb(v, torch.from_numpy(tb).cuda(), radius)
    ref = np.asarray(disk_mean_tb(v, tb.astype(np.float64), radius)).reshape(-1)
    assert np.allclose(out.cpu().numpy(), ref, rtol=1e-12, atol=1e-6)
