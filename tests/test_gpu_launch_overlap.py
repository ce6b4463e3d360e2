"""Kernels that start while the one before them ends, against the same kernels kept apart: with the
per-kernel timing on, an event stands between any two launches and nothing overlaps.  Every value
must be the same, from meshes of one CTA to several waves of them, along each chain of kernels
(gradients, boundary lifting, indicator, limiter, thermodynamics, chemistry, time step)."""
import numpy as np
import pytest

import cases
import workloads as W
from test_gpu_cta_shapes import NS, _box, _mixture
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


RUNS = [("box", 3, 3, (1, 1, 1), NS), ("box", 3, 3, (20, 17, 9), NS), ("box", 3, 4, (12, 10, 9), NS), ("box", 3, 7, (7, 5, 9), {}),
        ("box", 3, 7, (3, 2, 3), dict(alpha_max=0.5, positivity_eps=0.1, **NS)),
        ("box", 2, 3, (90, 61), dict(alpha_max=0.5, positivity_eps=0.1)),
        ("channel", 3, 3, (9, 8, 7), dict(bc_kind=[INFLOW, OUTFLOW], bc_prim=np.array([INFLOW_STATE] * 2), **NS)),
        ("channel", 3, 4, (3, 8, 7), dict(bc_kind=[NOSLIP, ISOTHERMAL], bc_prim=np.array([WALL] * 2), **NS)),
        ("mixture", 3, 4, (6, 8, 5), {}), ("mixture", 3, 3, (2, 4, 1), {}), ("chemistry", 3, 4, (6, 8, 5), {})]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kind,dim,N,shape,kw", RUNS)
def test_overlapped_launches_change_nothing(dg, precision, kind, dim, N, shape, kw):
    kw = dict(kw)
    if kind in ("mixture", "chemistry"):
        build = _mixture(shape)
        kinds, bcp = cases.mixture_bc(cases.mixture_ogrid(dg.dg_lgl_nodes(N)[0], *shape)[3])
        kw = dict(n_species=5, species=W.species_table(), volume_flux=1, bc_kind=kinds, bc_prim=bcp, alpha_max=0.5,
                  positivity_eps=0.1)
        if kind == "chemistry":
            kw["reactions"] = W.reaction_table()
    else:
        build = _box(shape, dim) if kind == "box" else _channel_builder(shape)
    xyz, nbr, face, w = build(dg.dg_lgl_nodes(N)[0])
    s = dg.Solver(dim, N, xyz, nbr, face, precision=precision, **kw)
    try:
        if kind == "channel":
            w = cases.perturbed_state(w, 5, amp=0.05)
        got = []
        for apart in (1, 0, 0):
            dg.dg_profile(s.ctx, apart)
            s.set_primitive(w)
            # (chemistry from a perturbed cold flow stays physical at a twentieth)
            t = s.step(4, cfl=0.01 if kind == "chemistry" else 0.2)
            u, _ = s.get_state()
            got.append((t, np.array(u)))
        for t, u in got[1:]:
            assert t == got[0][0] and np.array_equal(u, got[0][1])
        assert np.all(np.isfinite(got[0][1]))
    finally:
        s.close()


@pytest.mark.parametrize("batch,n_out,own_stream", [(1, 1, False), (200, 10, True), (4096, 10, False), (5000, 1, True)])
def test_overlapped_training_changes_nothing(dg, batch, n_out, own_stream):
    """Training iterations (two gathers into buffers that the last iteration read, gradient, Adam) with a
    synchronisation after each call and without any."""
    import torch
    g = torch.Generator().manual_seed(3)
    X = torch.randn((20000, 7), generator=g).cuda()
    Y = torch.randn((20000, n_out), generator=g).cuda()
    idx = torch.randint(0, 20000, (30, batch), generator=g).cuda()
    P0 = (0.3 * torch.randn((dg.dg_mlp_nparams(n_out),), generator=g)).cuda()
    stream = torch.cuda.Stream() if own_stream else None
    raw = stream.cuda_stream if own_stream else None
    got = []
    for apart in (True, False, False):
        P, m, v = P0.clone(), torch.zeros_like(P0), torch.zeros_like(P0)
        loss = torch.zeros((1,), dtype=torch.float64, device="cuda")
        ws = torch.empty((dg.dg_mlp_workspace_bytes(batch, n_out) // 4,), device="cuda")
        xb, yb = torch.empty((batch, 7), device="cuda"), torch.empty((batch, n_out), device="cuda")
        torch.cuda.synchronize()
        wait = torch.cuda.synchronize if apart else (lambda: None)
        for k in range(30):
            dg.dg_gather_rows(X, idx[k], xb, raw), wait()
            dg.dg_gather_rows(Y, idx[k], yb, raw), wait()
            dg.dg_mlp_train_step(P, m, v, xb, yb if n_out > 1 else yb.reshape(-1), k + 1, 1e-3, loss, ws, raw), wait()
        torch.cuda.synchronize()
        got.append((P, m, v, loss))
    for other in got[1:]:
        assert all(torch.equal(a, b) for a, b in zip(got[0], other))
    assert torch.isfinite(got[0][0]).all() and not torch.equal(got[0][0], P0)
