"""The mixed form's plain source with species that are absent, negative (overshoots next to a front)
or far below the usual range of concentrations, alone and beside usual ones in one warp: the source
and a step with its point-implicit terms against the oracle, and the time against the FP64
form's evaluation of the same state."""
import numpy as np
import pytest

import cases
import workloads as W
from test_gpu_chem_pairs import TOL, _solver, _source

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2511_17551_gb300 as dg
    dg.lib()
    return dg


def _absent(w):
    w[:, 0] = w[:, 3] = 0.0


def _one_left(w):
    w[:, [0, 2, 3, 4]] = 0.0


def _absent_in_places(w):
    w[:, 1, ::2] = w[:, 4, ::3] = 0.0


def _negative(w):
    w[:, 0] = -1e-6
    w[:, 2, ::3] *= -1e-3
    w[:, 3, ::5] = -1e-12


def _tiny(w):
    w[:, 0, ::2] = 3e-31
    w[:, 1, 1::2] = -2e-36
    w[:, 4, ::3] = 4e-40


def _all_of_it(w):
    rng = np.random.default_rng(2)
    kind = rng.integers(0, 5, (w.shape[0], 5, w.shape[2]))
    kind[:, 2] = 4
    r = w[:, :5]
    r[kind == 0] = 0.0
    r[kind == 1] *= -1e-4
    r[kind == 2] = 10.0 ** rng.uniform(-37, -16, (kind == 2).sum())


CHANGES = [_absent, _one_left, _absent_in_places, _negative, _tiny, _all_of_it]


@pytest.mark.parametrize("change", CHANGES)
@pytest.mark.parametrize("N,shape,hot", [(3, (2, 2, 2), (1.2, 2500.0)), (4, (3, 5, 3), (1.2, 9000.0)), (4, (2, 3, 2), None)])
def test_source(dg, change, N, shape, hot):
    import oracle
    s = _solver(dg, N, shape, hot, change)
    try:
        S, rho, T, _ = _source(dg, s)
        _, _, So = oracle.chem_eval(W.species_table(), W.reaction_table(), rho, T, 0.0)
        # below FP32's normal numbers: the rates are flushed at 2^-160 mol/(cm^3 s)
        err = np.abs(S - So) / (TOL * np.abs(So).sum(1, keepdims=True) + 2.0 ** -126)
        print("largest deviation in units of the bound", err.max(), "largest rate", np.abs(So).max())
        assert np.isfinite(S).all() and err.max() <= 1.0, err.max()
    finally:
        s.close()


@pytest.mark.parametrize("change", [_absent, _negative])
def test_step(dg, change):
    """One step long enough for the point-implicit factors of absent and negative species to count
    (changes that leave the flow smooth; the test checks that they do count)."""
    import oracle

    def build(x):
        xyz, nbr, face, w = cases.mixture_ogrid(x, hot=(1.2, 3000.0))
        change(w)
        return xyz, nbr, face, w

    kinds, bcp = cases.mixture_bc(cases.mixture_ogrid(oracle.lgl(3)[0])[3])
    p = cases.Pair(build, 3, 3, precision=1, n_species=5, species=W.species_table(), reactions=W.reaction_table(),
                   volume_flux=1, surface_flux=0, bc_kind=kinds, bc_prim=bcp)
    try:
        u = p.orc.prim_to_cons(p.mesh_o[3]).astype(np.float32).astype(np.float64)
        dt = 0.1 * p.orc.max_dt(u, 0.5)
        p.gpu.set_state(u)
        p.gpu.step(1, dt_fixed=dt)
        u_g, _ = p.gpu.get_state()
        u_r, _ = p.orc.step_rk(u, 1, dt_fixed=dt)
        err = cases.field_errors(u_g - u, u_r - u, 5, 3)
        # the increment is a sum of right-hand sides from FP32 states, whose temperature is good to 1e-6
        # (test_gpu_thermo_pairs); a rate changes by theta / T of that
        R = W.reaction_table()
        bar = 16.0 * cases.rounding_floor(p.orc, u) + 1e-6 * R[:, 18].max() / p.orc.temperature(u).max()
        rho, T = u[:, :5].transpose(0, 2, 1).reshape(-1, 5), p.orc.temperature(u).reshape(-1)
        om, _, S = oracle.chem_eval(W.species_table(), W.reaction_table(), rho, T, dt)
        odd = rho <= 0.0
        share = (np.abs(S - om)[odd] / (np.abs(om)[odd] + 1e-300)).max() if odd.any() else 1.0
        print("increment error", err, "bar", bar, "largest point-implicit reduction", share)
        assert np.all(err < bar), (err, bar)
        assert share > 1e-2
    finally:
        p.close()


def test_reactions_switched_off(dg):
    """A = 0: the source of the table without them, to the bit."""
    R = W.reaction_table()
    R0 = R.copy()
    R0[[2, 7], 16] = 0.0
    got = []
    for table in (R0, np.delete(R, [2, 7], 0)):
        x, _ = dg.dg_lgl_nodes(3)
        xyz, nbr, face, w = cases.mixture_ogrid(x, 2, 2, 2, hot=(1.2, 2500.0))
        kinds, bcp = cases.mixture_bc(w)
        s = dg.Solver(3, 3, xyz, nbr, face, n_species=5, species=W.species_table(), volume_flux=1, bc_kind=kinds,
                      bc_prim=bcp, precision=dg.DG_MIXED, reactions=table)
        try:
            s.set_primitive(w)
            got.append(_source(dg, s)[0])
        finally:
            s.close()
    assert np.array_equal(got[0], got[1]) and np.abs(got[0]).max() > 0.0


@pytest.mark.parametrize("change", [_absent_in_places, _negative])
def test_time_per_evaluation(dg, change):
    """Where every warp holds such nodes the mixed form still takes less than the FP64 form's time,
    about half of it (it evaluated them in FP64 behind the pairs, and took 1.1 times that time)."""
    import torch
    ms = []
    for precision in (dg.DG_FP64, dg.DG_MIXED):
        x, _ = dg.dg_lgl_nodes(4)
        xyz, nbr, face = W.ogrid_mesh(x, 16, 24, 8)
        w = W.mixture_primitive(xyz, rho=0.1, vel=(2400.0, 0.0, 0.0), T=300.0, seed=7, cylinder=0.5, hot=(1.2, 3000.0))
        kinds, bcp = cases.mixture_bc(w)
        change(w)
        s = dg.Solver(3, 4, xyz, nbr, face, n_species=5, species=W.species_table(), volume_flux=1, bc_kind=kinds,
                      bc_prim=bcp, precision=precision, reactions=W.reaction_table())
        try:
            s.set_primitive(w)
            u = torch.from_numpy(s.get_state()[0]).cuda()
            u = u.float() if precision == dg.DG_MIXED else u
            r = torch.empty_like(u)
            for _ in range(2):
                dg.dg_rhs(s.ctx, u, r)
            dg.dg_profile(s.ctx, 1)
            dg.dg_profile_read(s.ctx)
            for _ in range(10):
                dg.dg_rhs(s.ctx, u, r)
            ms.append(dg.dg_profile_read(s.ctx)["chem"][0])
        finally:
            s.close()
    print("FP64 and mixed form", ms)
    assert ms[1] < 0.8 * ms[0], ms
