"""The adjoint of steps whose tube area comes from the field's second
derivatives, of steps that retrace their neighbours, and of mixtures, against
the FP64 oracle's tape adjoint (which always retraces).

Bar, relative L2 over the nodes: 5e-3 for n_e and 1e-3 for T_e, those of the
single-precision path on these coarse coronae (a face that an FP32 stage
point crosses a step early moves a ray's gradient by its kink)."""
import numpy as np
import pytest

import corona_synth as cs
from test_gpu_curvature import corona
from test_gpu_parity import ctx, rt  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,lat,opts", [
    ((24, 16, 32), 0.2, dict(dtau=4e-3)),                          # nearly all steps from second derivatives
    ((24, 16, 32), 1.45, dict(dtau=8e-3)),                         # along the polar axis
    ((96, 64, 128), 0.2, dict(dtau=4e-3)),                         # a third of the steps retraced
    ((24, 16, 32), 0.2, dict(dtau=1.6e-2)),                        # all steps retraced
    ((24, 16, 32), 0.2, dict(dtau=4e-3, eps_mode=1, delta=1e-2)),  # offsets of a given length
    ((5, 3, 4), -0.5, dict(dtau=8e-3)),                            # a few large cells
    ((24, 16, 32), 0.2, dict(dtau=4e-3, s_mode=2)),
])
def test_adjoint_forms(rt, ctx, orc, shape, lat, opts):  # noqa: F811
    import torch
    g = corona(*shape)
    v = cs.View(0.4, lat, 6, 5, -1.7, 1.9, -1.5, 1.6)
    freqs = [90e6, 400e6]
    w = np.random.default_rng(3).normal(size=(2, v.ny, v.nx))
    grid = ctx.load(g)
    _, _, tape = ctx.trace_image_tape(grid, v, freqs, rt.options(precision=1, **opts))
    dne, dte = tape.backward(w)
    torch.cuda.synchronize()
    tape.free()
    gne, gte, _ = orc.backward(orc.grid_field(g), v, freqs, w.reshape(2, -1),
                               orc.default_options(tau_stop=30.0, **opts))
    for got, ref, bar in ((dne, gne, 5e-3), (dte, gte, 1e-3)):
        d = got.cpu().numpy().astype(np.float64) - ref
        rel = np.linalg.norm(d) / np.linalg.norm(ref)
        print(shape, opts, "relative L2", rel)
        assert rel <= bar, (shape, opts, rel)
