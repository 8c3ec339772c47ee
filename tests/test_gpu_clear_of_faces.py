"""The rule that takes a step's tube area from the field's second derivatives
holds where it says so: no neighbour of such a step leaves the cells of the
central ray's stage points.  A neighbour that is missed across a face leaves
the face's kink out of ln M, so ln S of the ray shows it against the FP64
oracle, which always retraces.

ln S bar as in test_gpu_curvature.py, 3e-4; one missed kink of these coronae
is several times that."""
import numpy as np
import pytest

import corona_synth as cs
from test_gpu_parity import compare, ctx, rt, run_gpu, run_oracle, spreads  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_nb,precision", [(4, 1), (8, 1), (4, 0)])
def test_steps_into_the_vacuum(rt, ctx, orc, n_nb, precision):  # noqa: F811
    """A low, dense corona left at all angles: on a ray's last step its second
    stage point may lie outside, and neighbours still inside, where the density
    falls off at half a force unit per step."""
    opts = dict(n_nb=n_nb, precision=precision, dtau=4e-3)
    g = cs.newkirk_grid(3, 16, 32, 1.05)
    v = cs.View(0.4, 0.2, 25, 23, -1.06, 1.06, -1.06, 1.06)
    freqs = [260e6, 330e6]
    gpu = run_gpu(rt, ctx, ctx.load(g), v, freqs, **opts)
    ref = run_oracle(orc, g, v, freqs, **opts)
    cond = spreads(orc, g, v, freqs, ref, **opts)
    bars = dict(lns_abs=3e-4) if precision else dict(exit_abs=1e-3, lns_abs=3e-4)
    rep = compare(gpu, ref, cond=cond, **bars, label=f"vacuum {opts}", min_well=0.5)
    assert rep["well_lns"] > 0.5


def share_of_second_derivatives(rt, ctx, grid, v, f_hz, opts):  # noqa: F811
    """The share of steps, from the 4th to the 60th of every ray, that take ln M
    from the second derivatives: there the offset's length is not in the
    arithmetic, so 1% more of it gives the same bits; retraced neighbours move."""
    key = "delta" if opts.get("eps_mode") else "eta"
    o = {"eta": 0.5, **opts, "max_steps": 60}
    pix = np.arange(v.nx * v.ny, dtype=np.int32)
    a, b = (ctx.trace_paths(grid, v, f_hz, pix, rt.options(**{**o, key: o[key] * c}), cap=61)[0] for c in (1.0, 1.01))
    same = [p["dlns_ds"][4:] == q["dlns_ds"][4:] for p, q in zip(a, b) if len(p["r"]) > 4]
    return float(np.concatenate(same).mean())


@pytest.mark.parametrize("n_nb,lat,f,opts", [
    (4, 0.3, 1, dict(eps_mode=1, delta=1e-3)),
    (8, 0.3, 1, dict(eps_mode=1, delta=3e-3)),
    (4, 1.5, 1, dict(eps_mode=1, delta=5e-3)),
    (8, -0.7, 1, dict(eps_mode=1, delta=4e-3, dtau=8e-3)),
    (4, 0.3, 1, dict(eta=0.1, dtau=1.5e-3)),
    (4, 0.3, 0, dict(eps_mode=1, delta=1e-2)),                # most of the corona lies within 256 offsets of the axis
    (4, 0.3, 0, dict(eps_mode=1, delta=2e-4)),                # small against the third stage's distance
    (4, 0.3, 0, dict(eta=0.1, dtau=8e-3)),
    (4, 0.3, 0, dict(eps_mode=1, delta=2e-2)),                # cells hardly wider than the offsets
])
def test_offsets_of_either_kind(rt, ctx, orc, n_nb, lat, f, opts):  # noqa: F811
    """Forward rows over the kinds of offset, each in the form (f: second
    derivatives, or every step retraced) that the rule gives it."""
    from test_gpu_curvature import corona
    opts = {"precision": 1, "dtau": 4e-3, "n_nb": n_nb, **opts}
    g = corona(64, 32, 64)
    v = cs.View(0.7, lat, 9, 7, -2.2, 2.6, -1.9, 2.1)
    freqs = [60e6, 300e6]
    grid = ctx.load(g)
    took = share_of_second_derivatives(rt, ctx, grid, v, freqs[0], opts)
    assert took > 0.5 if f else took < 0.05, (opts, took)
    gpu = run_gpu(rt, ctx, grid, v, freqs, **opts)
    ref = run_oracle(orc, g, v, freqs, **opts)
    cond = spreads(orc, g, v, freqs, ref, **opts)
    compare(gpu, ref, cond=cond, lns_abs=3e-4, label=f"offset {opts}", min_well=0.5)


@pytest.mark.parametrize("n_nb,delta", [(4, 3.5e-3), (8, 5e-3)])
def test_fixed_offset_at_turning_points(rt, ctx, orc, n_nb, delta):  # noqa: F811
    """Rays near the disk centre turn back where the force alone sets the
    chord's direction: neighbours at a fixed offset reach across radial faces
    there.  Cells of 0.13 R_sun, whose faces carry a strong kink, and many
    frequencies, so that some rays turn close to a face."""
    opts = dict(precision=1, dtau=8e-3, n_nb=n_nb, eps_mode=1, delta=delta)
    g = cs.newkirk_grid(16, 16, 32, 3.0)
    v = cs.View(0.7, 0.3, 12, 11, -0.1, 0.1, -0.1, 0.1)
    freqs = cs.log_freqs(32, 40e6, 160e6)
    grid = ctx.load(g)
    assert share_of_second_derivatives(rt, ctx, grid, v, freqs[0], opts) > 0.5
    gpu = run_gpu(rt, ctx, grid, v, freqs, **opts)
    ref = run_oracle(orc, g, v, freqs, **opts)
    cond = spreads(orc, g, v, freqs, ref, **opts)
    rep = compare(gpu, ref, cond=cond, lns_abs=3e-4, label=f"turning {opts}", min_well=0.5)
    assert rep["well_lns"] > 0.3
