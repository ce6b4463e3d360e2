"""A launch that the runtime refuses (on the legacy stream while a blocking stream is being captured) is
reported by that call and leaves nothing behind: the next calls succeed."""
import ctypes as C

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_refused_launch_is_reported_once():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2511_17551_gb300 as dg
    x, _ = dg.dg_lgl_nodes(3)
    xyz, nbr, face = W.box_mesh((2, 2), x, (-1.0,) * 2, (1.0,) * 2, periodic=True)
    s = dg.Solver(2, 3, xyz, nbr, face)
    try:
        X = torch.arange(70, dtype=torch.float32, device="cuda").reshape(10, 7)
        idx = torch.tensor([3, 1], device="cuda")
        out = torch.empty((2, 7), device="cuda")
        w = np.ones((4, 4, 16))
        torch.cuda.synchronize()
        rt = C.CDLL("libcudart.so.13")
        stream, graph = C.c_void_p(), C.c_void_p()
        assert rt.cudaStreamCreate(C.byref(stream)) == 0
        assert rt.cudaStreamBeginCapture(stream, 2) == 0
        with pytest.raises(dg.DgError) as e:
            dg.dg_gather_rows(X, idx, out)
        assert e.value.code == dg.DG_ECUDA
        left = rt.cudaPeekAtLastError()
        rt.cudaStreamEndCapture(stream, C.byref(graph))  # the refused launch has ended the capture
        assert left == 0
        rt.cudaGetLastError()
        assert rt.cudaStreamDestroy(stream) == 0
        s.set_primitive(w)
        dg.dg_gather_rows(X, idx, out)
        torch.cuda.synchronize()
        assert torch.equal(out, X[idx])
    finally:
        s.close()
