"""The path recorder's rays over warps: one ray to a warp up to full warps, the
same bits as the image's rays."""
import numpy as np
import pytest

import corona_synth as cs
from test_gpu_parity import ctx, rt, tiny  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 63, 608, 609, 1217, 20000])
@pytest.mark.parametrize("opts", [dict(n_nb=4), dict(n_nb=2), dict(s_mode=2)])
def test_rays_of_a_warp(rt, ctx, tiny, n, opts):  # noqa: F811
    import torch
    grid = ctx.load(tiny[0])
    v = cs.View(0.3, 0.2, 160, 130, -2.0, 2.0, -1.6, 1.7)
    o = rt.options(precision=1, dtau=8e-3, **opts)
    pix = np.random.default_rng(n).permutation(v.nx * v.ny)[:n].astype(np.int32)
    paths, tb, d = ctx.trace_paths(grid, v, 90e6, pix, o, cap=2)
    tb_i, d_i = ctx.trace_image(grid, v, [90e6], o, diag=True)
    torch.cuda.synchronize()
    idx = torch.from_numpy(pix).long().cuda()
    assert torch.equal(tb, tb_i.reshape(-1)[idx]) and torch.equal(d, d_i.reshape(-1, 7)[idx])
    steps = d.cpu().numpy()[:, 5]
    assert all(p["n_nodes"] == s + 1 or (s == 0 and p["n_nodes"] == 0) for p, s in zip(paths, steps))
