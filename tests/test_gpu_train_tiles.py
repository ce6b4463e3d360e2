"""Gradient and Adam kernels at batches around the 32-sample tiles and the 152-CTA grid and for
every kind of output count, against the oracle's FP64 back-propagation."""
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


@pytest.mark.parametrize("n_out", [1, 3, 10, 16])
@pytest.mark.parametrize("batch", [1, 31, 33, 64, 4864, 5000])
def test_gradient(env, batch, n_out):
    dg, oracle, torch = env
    rng = np.random.default_rng(batch + n_out)
    p = (0.3 * rng.normal(size=oracle.mlp_nparams(n_out))).astype(np.float32)
    X = rng.normal(size=(batch, 7)).astype(np.float32)
    t = rng.normal(size=(batch, n_out)).astype(np.float32)
    loss_o, g_o = oracle.mlp_loss_grad(p.astype(np.float64), X.astype(np.float64), t.astype(np.float64), n_out)
    P, Xd, td = (torch.from_numpy(a).cuda() for a in (p, X, t))
    grad = torch.empty_like(P)
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    ws = torch.empty(dg.dg_mlp_workspace_bytes(batch, n_out) // 4 + 1, dtype=torch.float32, device="cuda")
    ws[-1] = 5.0
    dg.dg_mlp_grad(P, Xd, td if n_out > 1 else td.reshape(-1), grad, loss, ws)
    torch.cuda.synchronize()
    g = grad.cpu().numpy().astype(np.float64)
    # FP32 sums of up to 5,000 terms, tree-like over tiles and CTAs: the bar of the other gradient tests
    assert np.linalg.norm(g - g_o) / np.linalg.norm(g_o) < 1e-5
    assert abs(loss.item() / loss_o - 1) < 1e-5
    assert ws[-1].item() == 5.0
    # the Adam step of the same gradient, twice: the same bits
    out = []
    for _ in range(2):
        q, m, v = P.clone(), torch.full_like(P, 1e-3), torch.full_like(P, 1e-5)
        dg.dg_mlp_train_step(q, m, v, Xd, td if n_out > 1 else td.reshape(-1), 7, 1e-3, loss, ws)
        torch.cuda.synchronize()
        out.append((q.cpu(), m.cpu(), v.cpu()))
    assert all(torch.equal(a, b) for a, b in zip(*out))
    m_o = 0.9 * 1e-3 + 0.1 * g_o
    v_o = 0.999 * 1e-5 + 0.001 * g_o * g_o
    step = 1e-3 * (m_o / (1 - 0.9 ** 7)) / (np.sqrt(v_o / (1 - 0.999 ** 7)) + 1e-8)
    assert np.abs(out[0][0].numpy() - (p - step)).max() < 1e-7 + 1e-4 * np.abs(step).max()
