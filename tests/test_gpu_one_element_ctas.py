"""FP64, 3D, N = 4: up to 152 elements the right-hand side takes one element a CTA, above that two.  The same
box alone and three times over in one mesh (on either side of that line) gives the same bits, and
a call below the line takes less time than one with two elements a CTA."""
import numpy as np
import pytest

import cases
import workloads as W
from test_gpu_cta_shapes import NS, _box
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


def _rhs(dg, mesh, copies, kw):
    """Right-hand side and state after two steps of `copies` separate copies of a mesh."""
    import torch
    xyz, nbr, face, w = mesh
    K = xyz.shape[0]
    nbr = np.concatenate([np.where(nbr >= 0, nbr + c * K, nbr) for c in range(copies)])
    s = dg.Solver(3, 4, np.tile(xyz, (copies, 1, 1)), nbr, np.tile(face, (copies, 1)), **kw)
    try:
        s.set_primitive(np.tile(w, (copies, 1, 1)))
        u = torch.from_numpy(s.get_state()[0]).cuda()
        r = torch.empty_like(u)
        dg.dg_rhs(s.ctx, u, r)
        dg.dg_sync(s.ctx)
        s.step(2, cfl=0.1)
        return r.cpu().numpy(), s.get_state()[0]
    finally:
        s.close()


@pytest.mark.parametrize("shape,kw", [((4, 5, 4), {}), ((4, 5, 4), NS), ((19, 4, 2), NS), ((5, 4, 4), dict(alpha_max=0.5, **NS)),
                                      ((5, 4, 4), dict(surface_flux=1)), ((5, 4, 4), dict(volume_flux=3, **NS)),
                                      ((5, 4, 4), dict(sutherland_s=0.4, sutherland_rt=0.9, **NS)),
                                      ((5, 4, 4), dict(bc_kind=[INFLOW, OUTFLOW], bc_prim=np.array([INFLOW_STATE] * 2), **NS)),
                                      ((5, 4, 4), dict(bc_kind=[NOSLIP, ISOTHERMAL], bc_prim=np.array([WALL] * 2), **NS))])
def test_both_shapes_give_the_same_bits(dg, shape, kw):
    x, _ = dg.dg_lgl_nodes(4)
    if "bc_kind" in kw:
        mesh = _channel_builder(shape)(x)
        mesh = (*mesh[:3], cases.perturbed_state(mesh[3], 5, amp=0.05))
    else:
        mesh = _box(shape, 3)(x)
    K = mesh[0].shape[0]
    assert K <= 152 < 2 * K
    one, two = _rhs(dg, mesh, 1, kw), _rhs(dg, mesh, 2, kw)
    for a, b in zip(one, two):
        assert np.isfinite(a).all() and np.abs(a).max() > 0.0
        assert np.array_equal(a, b[:K]) and np.array_equal(a, b[K:])


def test_time_below_the_line(dg):
    """150 elements take 0.73 of the time of 300, which are one CTA of two on each SM (with two elements a CTA
    both took the same)."""
    import time

    import torch
    x, _ = dg.dg_lgl_nodes(4)
    us = []
    for shape in ((5, 5, 6), (5, 10, 6)):
        xyz, nbr, face, w = _box(shape, 3)(x)
        s = dg.Solver(3, 4, xyz, nbr, face)
        try:
            s.set_primitive(w)
            u = torch.from_numpy(s.get_state()[0]).cuda()
            r = torch.empty_like(u)
            t = []
            for _ in range(8):
                dg.dg_sync(s.ctx)
                t0 = time.perf_counter()
                for _ in range(20):
                    dg.dg_rhs(s.ctx, u, r)
                dg.dg_sync(s.ctx)
                t.append((time.perf_counter() - t0) / 20)
            us.append(sorted(t)[1] * 1e6)
        finally:
            s.close()
    print("150 and 300 elements", us)
    assert us[0] < 0.94 * us[1], us
