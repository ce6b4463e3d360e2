"""The tcgen05 forward at the edges of its 256-row tiles (two rows per thread) and on buffers that
do not allow its 16-byte staging, against the oracle within its BF16 rounding model, as the other
forward tests (8 standard deviations per output)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_2511_17551_gb300 as dg
    dg.lib()
    return dg, oracle, torch


@pytest.mark.parametrize("n_out", [1, 10])
@pytest.mark.parametrize("n", [1, 127, 129, 255, 256, 257, 511, 1300])
@pytest.mark.parametrize("shift", [0, 1])
def test_forward_tile_edges(env, n_out, n, shift):
    dg, oracle, torch = env
    rng = np.random.default_rng(100 * n + n_out)
    p = (0.3 * rng.normal(size=oracle.mlp_nparams(n_out))).astype(np.float32)
    X = rng.normal(size=(n, 7)).astype(np.float32)
    P = torch.from_numpy(p).cuda()
    xb = torch.zeros(n * 7 + 1, device="cuda")  # shift: buffers 4 bytes off the 16-byte grid
    Xd = xb[shift:shift + n * 7].reshape(n, 7)
    Xd.copy_(torch.from_numpy(X))
    yb = torch.full((n * n_out + 9,), 7.0, device="cuda")
    y = yb[shift:shift + n * n_out].reshape(n, n_out)
    dg.dg_mlp_forward(P, Xd, y if n_out > 1 else y.reshape(-1), tensor_cores=2)
    torch.cuda.synchronize()
    y_o, sd = oracle.mlp_forward_sd(p.astype(np.float64), X.astype(np.float64), n_out)
    r = np.abs(y.cpu().numpy() - np.reshape(y_o, (n, n_out))) / np.reshape(sd, (n, n_out))
    assert r.max() <= 8.0, r.max()
    assert (yb[shift + n * n_out:] == 7.0).all() and (yb[:shift] == 7.0).all()


def test_forward_more_tiles_than_ctas(env):
    """Every CTA of the grid (1,216) takes several tiles, the last one ragged: row by row the same
    bits as a call on that row's tile alone."""
    dg, oracle, torch = env
    n = 256 * 2500 + 77
    g = torch.Generator("cuda").manual_seed(3)
    X = torch.randn((n, 7), generator=g, device="cuda")
    P = torch.from_numpy((0.3 * np.random.default_rng(4).normal(size=dg.dg_mlp_nparams(10))).astype(np.float32)).cuda()
    y = torch.empty((n, 10), device="cuda")
    dg.dg_mlp_forward(P, X, y, tensor_cores=2)
    for a, b in ((0, 256), (256 * 1215, 256 * 1217), (256 * 2432, 256 * 2433), (256 * 2499, n)):
        z = torch.empty((b - a, 10), device="cuda")
        dg.dg_mlp_forward(P, X[a:b].clone(), z, tensor_cores=2)
        torch.cuda.synchronize()
        assert torch.equal(y[a:b], z), (a, b)
