"""Sutherland's law in the kernels of the production flux pair (Ranocha, LLF): the degrees and
boundaries the other Sutherland tests leave out, against the oracle, and the same call through
the runtime-choice kernel's pair as a cross-check of the route."""
import numpy as np
import pytest

import cases
import workloads as W
from test_gpu_walls import INFLOW, INFLOW_STATE, ISOTHERMAL, NOSLIP, OUTFLOW, WALL, _channel_builder

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2511_17551_gb300 as dg
    dg.lib()
    return dg


@pytest.mark.parametrize("precision,tol", [(0, None), (1, 1e-5)])
@pytest.mark.parametrize("N,shape,where", [(2, (3, 2, 5), "box"), (7, (2, 2, 3), "box"), (3, (3, 4, 2), "inflow"),
                                           (4, (2, 3, 2), "walls")])
def test_cfl_steps_with_sutherland(dg, precision, tol, N, shape, where):
    """Two CFL steps (the wave speeds of the stage kernel weigh mu(T) too) and the step sizes."""
    if where == "box":
        kw = dict(W.supersonic_tgv_physics(), alpha_max=0.5)
        build = lambda x: cases.supersonic_tgv(x, None, warp=0.1, shape=shape)  # noqa: E731
    else:
        kw = dict(mu=0.02, Pr=0.72, sutherland_s=W.SUTHERLAND_S, sutherland_rt=0.9)
        build = _channel_builder(shape)
        kw["bc_kind"], kw["bc_prim"] = ([INFLOW, OUTFLOW], np.array([INFLOW_STATE] * 2)) if where == "inflow" else \
            ([NOSLIP, ISOTHERMAL], np.array([WALL] * 2))
    p = cases.Pair(build, 3, N, precision=precision, equations=1, **kw)
    try:
        w_o, w_g = (cases.perturbed_state(m[3], 5, amp=0.05) for m in (p.mesh_o, p.mesh_g))
        u_o = p.orc.prim_to_cons(w_o)
        p.gpu.set_primitive(w_g)
        t_g = p.gpu.step(2, cfl=0.3)
        u_g, _ = p.gpu.get_state()
        u_r, t_o = p.orc.step_rk(u_o, 2, cfl=0.3)
        err = cases.field_errors(u_g, u_r, 1, 3)
        bar = cases.fp64_bar(cases.step_floor(p.orc, u_o, 2, t_o / 2)) if tol is None else tol
        print(where, N, "steps error", err, "bar", bar)
        assert np.all(err < bar), (err, bar)
        assert abs(t_g / t_o - 1) < (1e-12 if tol is None else 1e-5)
    finally:
        p.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("N,shape", [(2, (3, 2, 5)), (3, (4, 3, 3)), (4, (3, 2, 3)), (7, (2, 2, 3))])
def test_production_and_runtime_choice_kernel_agree(dg, precision, N, shape):
    """Sutherland's law with LLF (the kernel of the production pair) and with HLLC (the runtime-choice kernel) on
    a flow whose traces agree at every face: both interface fluxes are then the flux of that trace, and
    the right-hand sides differ by roundings (16 times the oracle's floor)."""
    import torch
    kw = dict(W.supersonic_tgv_physics())
    got = []
    for sf in (0, 1):
        p = cases.Pair(lambda x: cases.supersonic_tgv(x, None, warp=0.1, shape=shape), 3, N, precision=precision, equations=1,
                       surface_flux=sf, **kw)
        try:
            u_o = p.orc.prim_to_cons(p.mesh_o[3])
            if precision:
                u_o = u_o.astype(np.float32).astype(np.float64)
            u = torch.from_numpy(u_o).cuda()
            u = u.float() if precision else u
            r = torch.empty_like(u)
            dg.dg_rhs(p.gpu.ctx, u, r)
            dg.dg_sync(p.gpu.ctx)
            got.append(r.double().cpu().numpy())
            if sf == 0:
                bar = 16.0 * cases.rounding_floor(p.orc, u_o, eps=2.0 ** (-24 if precision else -53))
        finally:
            p.close()
    err = cases.field_errors(got[1], got[0], 1, 3)
    print(N, precision, "difference of the routes", err, "bar", bar)
    assert np.all(err < bar), (err, bar)
