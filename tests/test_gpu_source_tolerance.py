"""The sampled check of the learned source with a tolerance beyond FP32's range, on states whose plain source is
zero: nothing but the floor decides, and every tile is accepted in both forms."""
import numpy as np
import pytest

import cases
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("tol", [0.1, 1e30, 1e300])
def test_zero_rates(precision, tol):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2511_17551_gb300 as dg
    x, _ = dg.dg_lgl_nodes(3)
    xyz, nbr, face, w = cases.mixture_ogrid(x, 3, 4, 2)
    w[:, [0, 1, 3, 4]] = 0.0  # one species, cold: no reaction has a rate that FP32 holds
    w[:, 8] = 250.0
    kinds, bcp = cases.mixture_bc(w)
    s = dg.Solver(3, 3, xyz, nbr, face, n_species=5, species=W.species_table(), volume_flux=1, bc_kind=kinds, bc_prim=bcp,
                  precision=precision, reactions=W.reaction_table())
    try:
        s.set_primitive(w)
        u = torch.from_numpy(s.get_state()[0]).cuda()
        u = u.float() if precision else u
        r = torch.empty_like(u)
        dg.dg_rhs(s.ctx, u, r)
        dg.dg_sync(s.ctx)
        assert np.abs(dg.dg_get_source(s.ctx, s.shape)[0]).max() < 1e-30
        p = (0.1 * np.random.default_rng(3).normal(size=dg.dg_mlp_nparams(10))).astype(np.float32)
        st = np.zeros(53)
        st[7:14], st[24:34], st[34], st[35] = [1, 1, 1, 1, 1, 5, 1000], 1.0, 1e-6, 1.0
        st[36:43], st[43:50], st[50:53] = -1e30, 1e30, [tol, 1e30, 1.0]
        dg.dg_set_surrogate(s.ctx, p, st, which=dg.DG_SURROGATE_SOURCE)
        dg.dg_rhs(s.ctx, u, r)
        accepted, recomputed = dg.dg_surrogate_stats(s.ctx, dg.DG_SURROGATE_SOURCE)
        assert recomputed == 0 and accepted == s.K * s.np, (accepted, recomputed)
    finally:
        s.close()
