"""Right-hand sides at element counts that leave the last CTA of every launch shape partly filled
(2 elements at N = 4, 1 or 2 for mixtures, 12 or 16 in 2D), for the production and the
runtime-choice pair, against the oracle."""
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


def _box(shape, dim):
    def build(x):
        xyz, nbr, face = W.box_mesh(shape, x, (-np.pi,) * dim, (np.pi,) * dim, periodic=True, warp=0.1 if dim == 3 else 0.0)
        rng = np.random.default_rng(11)
        w = np.zeros((xyz.shape[0], dim + 2, xyz.shape[2]))
        w[:, 0], w[:, 1 + dim] = 1.0, 2.0
        w[:, 1:1 + dim] = 0.3 * np.sin(xyz)
        return xyz, nbr, face, w * (1.0 + 0.05 * rng.uniform(-1, 1, w.shape))
    return build


def _mixture(shape):
    return lambda x: (lambda m: (*m[:3], cases.mixture_perturbed(m[3], 4)))(cases.mixture_ogrid(x, *shape))


NS = dict(equations=1, mu=0.02, Pr=0.72)
RUNS = [(3, 4, (3, 1, 3), NS), (3, 4, (5, 1, 1), dict(volume_flux=3, surface_flux=1)), (3, 4, (1, 1, 1), {}),
        (3, 4, (3, 3, 1), dict(alpha_max=0.5, **NS)), (3, 7, (3, 1, 1), {}), (3, 7, (1, 3, 1), dict(surface_flux=1)),
        (3, 3, (3, 3, 1), {}), (3, 2, (5, 3, 1), NS), (2, 3, (7, 5), dict(alpha_max=0.5)), (2, 3, (16, 1), dict(surface_flux=3)),
        (2, 4, (13, 1), {}), (2, 7, (7, 1), {}), (2, 2, (5, 5), {}),
        (3, 3, (3, 3, 3), "mixture"), (3, 4, (5, 3, 3), "mixture"), (3, 3, (1, 3, 1), "mixture_hllc"), (3, 4, (1, 1, 3), "mixture_hllc")]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("dim,N,shape,kw", RUNS)
def test_rhs(dg, precision, dim, N, shape, kw):
    import torch
    nsp = 1
    if isinstance(kw, str):
        nsp, build = 5, _mixture(shape)
        xo = dg.dg_lgl_nodes(N)[0]
        kinds, bcp = cases.mixture_bc(cases.mixture_ogrid(xo, *shape)[3])
        kw = dict(n_species=5, species=W.species_table(), volume_flux=1, surface_flux=1 if "hllc" in kw else 0,
                  bc_kind=kinds, bc_prim=bcp, alpha_max=0.5)
    else:
        build = _box(shape, dim)
    p = cases.Pair(build, dim, N, precision=precision, **kw)
    try:
        u_o = p.orc.prim_to_cons(p.mesh_o[3])
        real = torch.float32 if precision else torch.float64
        u = torch.from_numpy(u_o).cuda().to(real)
        r_o = p.orc.rhs(u.double().cpu().numpy())
        p.gpu.set_primitive(p.mesh_g[3])
        buf = torch.full((u.numel() + 64,), 3.0, dtype=real, device="cuda")
        r = buf[:u.numel()].reshape(u.shape)
        dg.dg_rhs(p.gpu.ctx, u, r)
        dg.dg_sync(p.gpu.ctx)
        err = cases.field_errors(r.double().cpu().numpy(), r_o, nsp, dim)
        # FP64: 1e-12 or 16 one-ulp floors of this input; mixed: 16 FP32 floors
        bar = cases.fp64_bar(cases.rounding_floor(p.orc, u_o, eps=2.0 ** -53)) if not precision else \
            np.maximum(16.0 * cases.rounding_floor(p.orc, u_o), 1e-6)
        print("error", err, "bar", bar)
        assert np.all(err < bar), (err, bar)
        assert (buf[u.numel():] == 3.0).all()
    finally:
        p.close()
