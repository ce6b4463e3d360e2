"""The FP64 right-hand sides' own reciprocal and square root (RealOps<double> of dg_kernels.cuh), in a kernel
of this test's own, against the correctly rounded ones over the range of FP64's normal numbers, and
what they give for zeros, infinities, NaN and at the ends of the range."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <stdint.h>
#include "dg_kernels.cuh"
__global__ void f(const double* x, double* r, int64_t n) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  double a, b;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(a) : "d"(x[i]));
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(b) : "d"(x[i]));
  r[6 * i + 0] = dgk::RealOps<double>::rcp(x[i]);
  r[6 * i + 1] = __drcp_rn(x[i]);
  r[6 * i + 2] = dgk::RealOps<double>::sqrt_(x[i]);
  r[6 * i + 3] = __dsqrt_rn(x[i]);
  r[6 * i + 4] = a;
  r[6 * i + 5] = b;
}
extern "C" int run(const double* x, double* r, long long n) {
  f<<<(unsigned)((n + 255) / 256), 256>>>(x, r, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_17551_gb300 import build
    d = tmp_path_factory.mktemp("fp64")
    (d / "f.cu").write_text(SOURCE)
    subprocess.check_call([build._nvcc()] + build.ARCH + build.FLAGS + ["-I", build.CSRC, "-shared", "-o", str(d / "f.so"),
                                                                       str(d / "f.cu")])
    fn = C.CDLL(str(d / "f.so")).run
    fn.argtypes = [C.c_void_p, C.c_void_p, C.c_longlong]

    def call(x):
        t = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        r = torch.empty((len(x), 6), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert fn(t.data_ptr(), r.data_ptr(), len(x)) == 0
        return r.cpu().numpy()
    return call


def _ulps(a, b):
    return np.abs(a.view(np.int64) - b.view(np.int64))


def test_normal_numbers(evaluate):
    """Householder's step of order three leaves the cube of the approximation's error, and the two
    functions one rounding (reciprocal) or one and a half (square root): within a unit."""
    rng = np.random.default_rng(4)
    n = 4_000_000
    bits = (rng.integers(1, 2045, n).astype(np.uint64) << np.uint64(52)) | rng.integers(0, 2 ** 52, n).astype(np.uint64)
    x = bits.view(np.float64)
    edge = 2.0 ** np.arange(-1022, 1022, dtype=np.float64)
    x = np.concatenate([x, 1.0 + rng.random(n), edge, np.nextafter(edge, 0)[1:], np.nextafter(edge, np.inf)])
    r = evaluate(np.concatenate([x, -x]))
    m = len(x)
    assert np.array_equal(r[m:, 0], -r[:m, 0]) and np.isnan(r[m:, 2]).all()
    ok = np.abs(r[:m, 1]) >= 2.0 ** -1022  # a normal reciprocal
    err = _ulps(r[:m, 0], r[:m, 1])[ok].max(), _ulps(r[:m, 2], r[:m, 3]).max()
    exact = np.longdouble(1) / x.astype(np.longdouble)
    start = np.abs(r[:m, 4].astype(np.longdouble) / exact - 1)[ok].max(), \
        np.abs(r[:m, 5].astype(np.longdouble) * np.sqrt(x.astype(np.longdouble)) - 1).max()
    print("units in the last place", err, "start values: log2 of the relative error", np.log2(np.float64(start)))
    assert max(err) <= 1
    assert (r[:m, 0][~ok] == 0.0).all()  # below the normal numbers: zero


def test_special_values(evaluate):
    tiny, inf, nan = 2.0 ** -1022, np.inf, np.nan
    x = np.array([0.0, -0.0, inf, -inf, nan, -nan, tiny, -tiny, 5e-324, -5e-324, tiny * (1 - 2.0 ** -52), 1.7976931348623157e308, 1.0, 4.0])
    r = evaluate(x)
    rcp = [inf, -inf, 0.0, -0.0, nan, nan, 2.0 ** 1022, -2.0 ** 1022, inf, -inf, inf, 0.0, 1.0, 0.25]
    root = [0.0, -0.0, inf, nan, nan, nan, 2.0 ** -511, nan, 5e-324, None, tiny * (1 - 2.0 ** -52), np.sqrt(x[11]), 1.0, 2.0]
    for i in range(len(x)):
        assert np.array_equal(r[i, 0], rcp[i], equal_nan=True) and (np.isnan(rcp[i]) or np.signbit(r[i, 0]) == np.signbit(rcp[i])), (x[i], r[i])
        # subnormal arguments come back as they are, of either sign: zero for what follows
        want = x[i] if root[i] is None else root[i]
        assert np.array_equal(r[i, 2], want, equal_nan=True) and (np.isnan(want) or np.signbit(r[i, 2]) == np.signbit(want)), (x[i], r[i])
