"""The beam convolution is linear down to the smallest floats: a map in units
2^k times larger gives the same bits 2^-k times smaller."""
import numpy as np
import pytest

import corona_synth as cs
from test_gpu_maps import maps
from test_gpu_parity import ctx, rt  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [-104, -60, -40, 60, 100, 110, 120])
@pytest.mark.parametrize("baseline", [15e3, 2e3, 2e5])
def test_beam_of_any_unit(rt, ctx, baseline, k):  # noqa: F811
    import torch
    v = cs.View(0.0, 0.0, 210, 90, -2.1, 2.1, -0.9, 0.9)
    f = [60e6, 400e6]
    tb = torch.from_numpy(maps(2, 90, 210)).cuda()
    out = ctx.beam_convolve(v, tb, f, baseline)
    small = ctx.beam_convolve(v, tb * 2.0 ** -k, f, baseline)
    assert torch.equal(small, out * 2.0 ** -k)


def test_beam_of_mixed_sizes(rt, ctx):  # noqa: F811
    """Values whose sums take the FP64 loop beside ordinary ones: outputs that no large value reaches
    keep their bits."""
    import torch
    v = cs.View(0.0, 0.0, 400, 90, -4.0, 4.0, -0.9, 0.9)
    tb = torch.from_numpy(maps(1, 90, 400)).cuda()
    base = ctx.beam_convolve(v, tb, [60e6], 1e3)
    t = tb.clone()
    t[0, 40, 390] = 2.0 ** 90
    out = ctx.beam_convolve(v, t, [60e6], 1e3)
    assert torch.isfinite(out).all()
    same = out == base
    from oracle import beam_sigma_pixels
    hw = int(np.ceil(4 * beam_sigma_pixels(v, 60e6, 1e3)))
    assert 64 < hw < 300 and same[0, :, :390 - hw].all() and not same[0, 40, 390 - hw // 2:].any()


def test_beam_of_nan(rt, ctx):  # noqa: F811
    import torch
    v = cs.View(0.0, 0.0, 210, 90, -2.1, 2.1, -0.9, 0.9)
    out = ctx.beam_convolve(v, torch.full((2, 90, 210), float("nan"), device="cuda"), [60e6, 400e6], 15e3)
    assert torch.isnan(out).all()
