"""The mixed form's temperature solve (FP32 Newton, residual in double-FP32 pairs) against the
oracle's Newton iteration on the same FP32-valued states: ragged element counts, cold and hot
states, densities on both sides of the pairs' range, and energies outside the clamp."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu

# the temperature coefficients of a node carry about ten FP32 roundings (mass fractions, products,
# sums), 2^-24 each of e(T) - e(0): 6e-7 of T
TOL = 1e-6


@pytest.fixture(scope="module")
def dg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2511_17551_gb300 as dg
    dg.lib()
    return dg


@pytest.mark.parametrize("scale", [1.0, 1e-8, 1e-13, 1e3])
@pytest.mark.parametrize("N,shape,hot", [(3, (1, 3, 2), None), (4, (3, 5, 3), (1.2, 9000.0)), (4, (2, 7, 2), (1.2, 2500.0))])
def test_mixed_temperature(dg, N, shape, hot, scale):
    import oracle
    import workloads as W
    x, _ = dg.dg_lgl_nodes(N)
    xyz, nbr, face, w = cases.mixture_ogrid(x, *shape, hot=hot)
    w[:, :5] *= scale
    kinds, bcp = cases.mixture_bc(w)
    sp = W.species_table()
    s = dg.Solver(3, N, xyz, nbr, face, n_species=5, species=sp, volume_flux=1, bc_kind=kinds, bc_prim=bcp,
                  precision=dg.DG_MIXED)
    xo, _ = oracle.lgl(N)
    mesh = cases.mixture_ogrid(xo, *shape, hot=hot)
    o = oracle.Oracle(3, N, *mesh[:3], n_species=5, species=sp, volume_flux=1, bc_kind=kinds, bc_prim=bcp)
    try:
        u = o.prim_to_cons(w).astype(np.float32)
        u[::2, 8, 1] *= 4.0     # far hotter: clamped where the energy passes e(1e4 K)
        u[::2, 8, 3] -= np.float32(0.999) * np.abs(u[::2, 8, 3])  # far colder: clamped to 200 K
        u64 = u.astype(np.float64)
        T_o = o.temperature(u64)
        s.set_state(u64)
        T = dg.dg_get_temperature(s.ctx, (s.K, s.np))  # from the cold start
        T2 = dg.dg_get_temperature(s.ctx, (s.K, s.np))  # from the cached temperature
        for t in (T, T2):
            err = np.abs(t / T_o - 1)
            print("scale", scale, "max", err.max())
            assert err.max() < TOL, err.max()
    finally:
        s.close()
