"""The step-wise tube area from the field's second derivatives (steps clear of
the cells' faces) and from retraced neighbours (the others, and every step
where the rule on cell widths and step length says so), against the FP64
oracle, which always retraces: T_b, exit points and ln S of the rays that are
well-conditioned for each, and the path recorder bit for bit.

ln S bar 3e-4: the form leaves out (eps / rho)^2 <= 1.6e-5 of each step's ln M
and third orders of at most 1e-9, and the FP32 paths are held to 1e-4
elsewhere.  The
plain form's paths drift by the rounding of their steps: its exit points and
ln S have the bars of test_tiny_full_map_plain, 1e-3 R_sun and 1e-2."""
import math

import numpy as np
import pytest

import corona_synth as cs
from test_gpu_parity import compare, ctx, rt, run_gpu, run_oracle, spreads  # noqa: F401

pytestmark = pytest.mark.gpu


def corona(n_r, n_t, n_p, r_max=4.0):
    g = cs.newkirk_grid(n_r, n_t, n_p, r_max)
    R, T, P = np.meshgrid(g.r, g.theta, g.phi, indexing="ij")
    return cs.Grid(g.r, g.theta, g.phi, g.ne * (1 + 0.3 * np.sin(2 * T) * np.cos(P - 0.5) * np.exp(-(R - 1))),
                   g.te * (1 + 0.2 * np.cos(T) * np.sin(2 * P)))


@pytest.mark.parametrize("shape,lat,opts", [
    ((64, 32, 64), 0.3, dict(n_nb=4)),                                  # few steps near a face
    ((64, 32, 64), 0.3, dict(n_nb=8, precision=0)),
    ((64, 32, 64), 1.5, dict(n_nb=4, precision=0)),                     # rays along the polar axis
    ((64, 32, 64), 1.5, dict(n_nb=8, dtau=8e-3)),
    ((128, 96, 192), 0.3, dict(n_nb=8)),                                # about a quarter of the steps
    ((128, 96, 192), 0.3, dict(n_nb=4, dtau=6e-3)),                     # about half
    ((128, 96, 192), 0.3, dict(n_nb=4, dtau=1.2e-2)),                   # the rule's other side
    ((9, 4, 5), -0.4, dict(n_nb=4, dtau=8e-3)),                         # cells far larger than a step
    ((9, 4, 5), -0.4, dict(n_nb=8, dtau=1.3e-2)),                       # a step too long for the form
    ((64, 32, 64), 0.3, dict(n_nb=4, eps_mode=1, delta=2e-4)),          # offsets of a given length
    ((64, 32, 64), 0.3, dict(n_nb=8, eps_mode=1, delta=2e-2)),
    ((64, 32, 64), 0.3, dict(n_nb=4, eta=2.0)),
])
def test_tube_area_forms(rt, ctx, orc, shape, lat, opts):  # noqa: F811
    import torch
    opts = {"precision": 1, "dtau": 4e-3, **opts}
    g = corona(*shape)
    v = cs.View(0.7, lat, 9, 7, -2.2, 2.6, -1.9, 2.1)
    freqs = [60e6, 300e6]
    grid = ctx.load(g)
    gpu = run_gpu(rt, ctx, grid, v, freqs, **opts)
    ref = run_oracle(orc, g, v, freqs, **opts)
    cond = spreads(orc, g, v, freqs, ref, **opts)
    bars = dict(lns_abs=3e-4) if opts["precision"] else dict(exit_abs=1e-3, lns_abs=1e-2)
    compare(gpu, ref, cond=cond, **bars, label=f"{shape} {opts}", min_well=0.5)
    o = rt.options(**opts)
    pix = np.arange(v.nx * v.ny, dtype=np.int32)
    _, tb_p, d_p = ctx.trace_paths(grid, v, freqs[0], pix, o, cap=4)
    tb_i, d_i = ctx.trace_image(grid, v, freqs[:1], o, diag=True)
    torch.cuda.synchronize()
    assert torch.equal(tb_p, tb_i.reshape(-1)) and torch.equal(d_p, d_i.reshape(-1, 7))
    assert math.isfinite(float(tb_p.sum()))
