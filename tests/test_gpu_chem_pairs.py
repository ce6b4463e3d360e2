"""The mixed form's plain source, evaluated in double-FP32 pairs (dg_dd.cuh) and rounded to
FP32, against the oracle's FP64 source at the GPU's own temperatures."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu

# per node: half an FP32 unit of the largest component, and as much again for the pairs
TOL = 2.0 ** -23


@pytest.fixture(scope="module")
def dg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2511_17551_gb300 as dg
    dg.lib()
    return dg


def _solver(dg, N, shape, hot, change):
    import workloads as W
    x, _ = dg.dg_lgl_nodes(N)
    xyz, nbr, face, w = cases.mixture_ogrid(x, *shape, hot=hot)
    kinds, bcp = cases.mixture_bc(w)
    change(w)
    s = dg.Solver(3, N, xyz, nbr, face, n_species=5, species=W.species_table(), volume_flux=1, surface_flux=0,
                  bc_kind=kinds, bc_prim=bcp, precision=dg.DG_MIXED, reactions=W.reaction_table())
    s.set_primitive(w)
    return s


def _source(dg, s):
    """(S [n][5], rho_s [n][5], T [n]) of the current state rounded to FP32."""
    import torch
    u = torch.from_numpy(s.get_state()[0]).cuda().float()
    r = torch.empty_like(u)
    s.set_state(u.double())
    dg.dg_get_temperature(s.ctx, (s.K, s.np))  # from the cold start
    dg.dg_rhs(s.ctx, u, r)
    dg.dg_sync(s.ctx)
    S, flags, _ = dg.dg_get_source(s.ctx, s.shape)
    T = dg.dg_get_temperature(s.ctx, (s.K, s.np)).reshape(-1)
    rho = u[:, :5].double().cpu().numpy().transpose(0, 2, 1).reshape(-1, 5)
    return S.transpose(0, 2, 1).reshape(-1, 5), rho, T, flags


def _none(w):
    pass


def _zero_species(w):  # concentrations the pairs do not hold: the FP64 evaluation
    w[:, 0] = 0.0
    w[::2, 3] = 0.0


def _some_tiny(w):  # both evaluations in one warp
    w[:, 1, ::3] = 1e-25


def _dense(w):
    w[:, :5] *= 200.0


def _thin(w):
    w[:, :5] *= 1e-7


@pytest.mark.parametrize("change", [_none, _zero_species, _some_tiny, _dense, _thin])
@pytest.mark.parametrize("N,shape,hot", [(3, (2, 2, 2), (1.2, 2500.0)), (4, (3, 5, 3), (1.2, 9000.0)),
                                         (4, (2, 3, 2), None)])
def test_mixed_source_is_the_rounded_fp64_source(dg, change, N, shape, hot):
    import oracle
    import workloads as W
    s = _solver(dg, N, shape, hot, change)
    try:
        S, rho, T, _ = _source(dg, s)
        _, _, So = oracle.chem_eval(W.species_table(), W.reaction_table(), rho, T, 0.0)
        scale = np.abs(So).sum(1, keepdims=True)
        # below the range of FP32 normal numbers a unit in the last place is 2^-149
        err = np.abs(S - So) / (TOL * scale + 2.0 ** -148)
        print("largest deviation in units of the bound", err.max(), "largest rate", np.abs(So).max())
        assert np.isfinite(S).all() and err.max() <= 1.0, err.max()
    finally:
        s.close()


def test_rejected_tiles_reproduce_the_mixed_plain_source_bitwise(dg):
    s = _solver(dg, 3, (3, 4, 2), (1.2, 2500.0), _some_tiny)
    try:
        S_plain, _, _, flags = _source(dg, s)
        assert (flags == 255).all()
        p = (0.3 * np.random.default_rng(3).normal(size=dg.dg_mlp_nparams(10))).astype(np.float32)
        st = np.zeros(53)
        st[7:14], st[24:34], st[34], st[35] = 1.0, 1.0, 1e2, 1e3
        st[36:43], st[43:50], st[50:52] = 1e30, -1e30, 1e30
        dg.dg_set_surrogate(s.ctx, p, st, which=dg.DG_SURROGATE_SOURCE)  # an empty trust box
        S_box, _, _, flags = _source(dg, s)
        assert (flags == 1).all() and np.array_equal(S_box, S_plain)
        dg.dg_set_source_refresh(s.ctx, 1)  # a refresh takes the plain source too
        S_ref, _, _, flags = _source(dg, s)
        assert (flags == 3).all() and np.array_equal(S_ref, S_plain)
    finally:
        s.close()
