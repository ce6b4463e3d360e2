"""The split of an FP64 state into the two FP32 parts of the mixed form and back, against numpy's
conversions: every class of value (zeros, subnormals, the ends of FP32's range, ties, values exact in
FP32), element counts with and without a last odd value, aligned and unaligned buffers.  numpy and
the device round to nearest even, so the values are equal to the bit."""
import numpy as np
import pytest

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


def _values(n, seed):
    rng = np.random.default_rng(seed)
    f = np.float64(np.float32(rng.standard_normal(n) * 10.0 ** rng.integers(-36, 37, n)))
    ulp = np.float64(np.spacing(np.abs(f).astype(np.float32)))
    x = f + ulp * rng.choice([0.0, 0.5, -0.5, 0.25, 0.5000000001, 0.4999999999, 0.123456789], n)
    some = np.array([0.0, -0.0, 2.0 ** -126, 2.0 ** -127, -(2.0 ** -149), 1e-46, 1e-300, 5e-324, 2.0 ** 127 * (2 - 2.0 ** -23),
                     -1.0, 1 + 2.0 ** -24, 1 + 3 * 2.0 ** -24, 1 + 2.0 ** -52, 2 - 2.0 ** -52, 2.0 ** -126 * (1 - 2.0 ** -30),
                     2.0 ** -126 * (1 + 2.0 ** -30), 1e-20, 2.0 ** -103 * (1 + 2.0 ** -40)])
    x[rng.integers(0, n, 4 * len(some))] = np.tile(some, 4)
    return x


@pytest.mark.parametrize("shape,off", [((8, 1), 0), ((7, 1), 0), ((7, 1), 1), ((90, 31), 0), ((8, 3), 1)])
def test_set_and_get_state(dg, shape, off):
    import torch
    N = 2  # nine nodes and four fields: an odd element count gives pairs that cross the fields
    xi = dg.dg_lgl_nodes(N)[0]
    xyz, nbr, face = W.box_mesh(shape, xi, (-np.pi,) * 2, (np.pi,) * 2, periodic=True)
    s = dg.Solver(2, N, xyz, nbr, face, precision=dg.DG_MIXED)
    try:
        x = _values(xyz.shape[0] * 4 * 9, 3).reshape(-1, 4, 9)
        buf = torch.empty(x.size + 2, dtype=torch.float64, device="cuda")
        src = buf[off:off + x.size].reshape(x.shape)
        src.copy_(torch.from_numpy(x))
        torch.cuda.synchronize()
        dg.dg_set_state(s.ctx, src, 0.0)
        hi = x.astype(np.float32)
        lo = (x - hi.astype(np.float64)).astype(np.float32)
        want = hi.astype(np.float64) + lo.astype(np.float64)
        out = torch.full((x.size + 2,), 7.0, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        dst = out[off:off + x.size].reshape(x.shape)
        dg.dg_get_state(s.ctx, dst)
        got = dst.cpu().numpy()
        assert np.array_equal(got, want) and np.array_equal(np.signbit(got), np.signbit(want))
        assert (out[off + x.size:] == 7.0).all() and (out[:off] == 7.0).all()
    finally:
        s.close()


def test_set_primitive_at_rest_and_tiny(dg):
    """Primitive to split conserved state, with zero and subnormal velocities among the values."""
    rng = np.random.default_rng(8)
    xi = dg.dg_lgl_nodes(3)[0]
    xyz, nbr, face = W.box_mesh((5, 3), xi, (-np.pi,) * 2, (np.pi,) * 2, periodic=True)
    w = 1.0 + 0.5 * rng.uniform(-1, 1, (15, 4, 16))
    w[:5, 1:3] = 0.0
    w[5:8, 1:3] = 1e-42 * rng.uniform(-1, 1, (3, 2, 16))
    s = dg.Solver(2, 3, xyz, nbr, face, precision=dg.DG_MIXED)
    try:
        s.set_primitive(w)
        u, _ = s.get_state()
        m = w[:, 0:1] * w[:, 1:3]
        hi = m.astype(np.float32)
        want = hi.astype(np.float64) + (m - hi.astype(np.float64)).astype(np.float32).astype(np.float64)
        assert np.array_equal(np.asarray(u)[:, 1:3], want)
    finally:
        s.close()
