"""Domain integrals (Eqs. TGV_KE, TGV_SD, TGV_DD) at element counts around the diagnostics kernel's
groups and for every degree and dimension, against plain numpy sums over the oracle's metric
terms and derivatives."""
import numpy as np
import pytest

import cases
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2511_17551_gb300 as dg
    dg.lib()
    return dg


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("dim,N,shape", [(3, 2, (2, 3, 5)), (3, 3, (5, 1, 1)), (3, 4, (3, 1, 1)), (3, 7, (3, 2, 1)),
                                         (3, 3, (13, 15, 13)), (2, 2, (5, 6)), (2, 3, (17, 1)), (2, 7, (3, 3)), (2, 4, (1, 1))])
def test_integrals(dg, precision, dim, N, shape):
    import oracle
    x, wq = oracle.lgl(N)
    xg, _ = dg.dg_lgl_nodes(N)
    lo, hi = (-np.pi,) * dim, (np.pi,) * dim
    xyz, nbr, face = W.box_mesh(shape, xg, lo, hi, periodic=True, warp=0.1 if dim == 3 else 0.0)
    rng = np.random.default_rng(7)
    K, npn = xyz.shape[0], (N + 1) ** dim
    u = np.zeros((K, dim + 2, npn))
    u[:, 0] = 1.0 + 0.1 * rng.uniform(-1, 1, (K, npn))
    u[:, 1:1 + dim] = rng.uniform(-1, 1, (K, dim, npn))
    u[:, 1 + dim] = 20.0 + rng.uniform(-1, 1, (K, npn))
    u = u.astype(np.float32).astype(np.float64)
    s = dg.Solver(dim, N, xyz, nbr, face, precision=precision)
    try:
        s.set_state(u)
        got = s.diagnostics()
        Ja, iJ = np.zeros((K, dim, dim, npn)), np.zeros((K, npn))
        dg.dg_get_metrics(s.ctx, Ja, iJ)
    finally:
        s.close()
    # derivative matrix of the Lagrange basis on the LGL nodes
    V = np.stack([np.polynomial.legendre.Legendre.basis(j)(x) for j in range(N + 1)], 1)
    dV = np.stack([np.polynomial.legendre.Legendre.basis(j).deriv()(x) if j else 0 * x for j in range(N + 1)], 1)
    D = dV @ np.linalg.inv(V)
    rho, E = u[:, 0], u[:, 1 + dim]
    v = u[:, 1:1 + dim] / rho[:, None]
    grid = (N + 1,) * dim
    vg = v.reshape((K, dim) + grid)
    dv = np.stack([np.moveaxis(np.moveaxis(vg, -1 - d, -1) @ D.T, -1, -1 - d).reshape(K, dim, npn)
                   for d in range(dim)], 1)  # [K][d][a][np]
    g = np.einsum("kdxn,kdan,kn->kaxn", Ja, dv, iJ)
    w = np.ones(1)
    for _ in range(dim):
        w = np.multiply.outer(w, wq).reshape(-1)
    dVol = w / iJ
    p = 0.4 * (E - 0.5 * rho * (v ** 2).sum(1))
    if dim == 3:
        w2 = (g[:, 2, 1] - g[:, 1, 2]) ** 2 + (g[:, 0, 2] - g[:, 2, 0]) ** 2 + (g[:, 1, 0] - g[:, 0, 1]) ** 2
    else:
        w2 = (g[:, 1, 0] - g[:, 0, 1]) ** 2
    div = np.einsum("kaan->kn", g)
    vol = dVol.sum()
    want = np.array([(dVol * 0.5 * rho * (v ** 2).sum(1)).sum() / vol, (dVol * 0.5 * rho * w2).sum() / vol,
                     (-dVol * rho * (np.log(p) - 1.4 * np.log(rho)) / 0.4).sum(), (dVol * rho).sum(), (dVol * E).sum(), vol,
                     (dVol * div ** 2).sum() / vol, (dVol * w2).sum() / vol])
    # sums of up to 160,000 FP64 terms of one sign (the entropy's change sign mildly): 1e-12
    assert np.abs(got / want - 1).max() < 1e-12, got / want - 1
