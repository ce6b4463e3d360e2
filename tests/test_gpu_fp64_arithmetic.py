"""The FP64 right-hand sides' own reciprocal, square root and logarithmic means against the oracle: states
scaled far from one (the range of the approximations they start from) and neighbouring values
on both sides of the line between the series and the logarithm (f^2 = 1e-4, a ratio of 1.02)."""
import numpy as np
import pytest

import cases
from test_gpu_cta_shapes import NS, _box

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2511_17551_gb300 as dg
    dg.lib()
    return dg


@pytest.mark.parametrize("N,scale,amp,kw", [
    (3, 1e-140, 0.05, {}), (3, 1e140, 0.05, {}), (4, 1e-140, 0.3, dict(surface_flux=1)), (7, 1e140, 0.3, {}),
    (3, 1.0, 0.004, NS), (3, 1.0, 0.01, NS), (4, 1.0, 0.02, dict(alpha_max=0.5)), (2, 1.0, 0.6, NS), (3, 1.0, 0.0, {})])
def test_rhs_fp64(dg, N, scale, amp, kw):
    import torch
    p = cases.Pair(_box((3, 2, 3), 3), 3, N, **kw)
    try:
        w = p.mesh_o[3].copy()
        w[:, 0], w[:, 4] = 1.0, 2.0
        w *= 1.0 + amp * np.random.default_rng(5).uniform(-1, 1, w.shape)
        u_o = p.orc.prim_to_cons(w) * scale
        u = torch.from_numpy(u_o).cuda()
        r = torch.empty_like(u)
        dg.dg_rhs(p.gpu.ctx, u, r)
        dg.dg_sync(p.gpu.ctx)
        r_o = p.orc.rhs(u_o)
        err = cases.field_errors(r.cpu().numpy() / scale, r_o / scale, 1, 3)
        bar = cases.fp64_bar(cases.rounding_floor(p.orc, u_o, eps=2.0 ** -53))
        print("error", err, "bar", bar)
        assert np.all(err < bar), (err, bar)
    finally:
        p.close()
