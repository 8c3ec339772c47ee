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
