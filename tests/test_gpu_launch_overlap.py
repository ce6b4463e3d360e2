"""Kernels that start while the one before them ends, against the same kernels kept apart: with the
per-kernel timing on, an event stands between any two launches and nothing overlaps.  Every value
must be the same, from meshes of one CTA to several waves of them, along each chain of kernels
(gradients, boundary lifting, indicator, limiter, thermodynamics, chemistry, time step)."""
import numpy as np
import pytest

import cases
import workloads as W
from test_gpu_cta_shapes import NS, _box, _mixture
from test_gpu_walls import INFLOW, INFLOW_STATE, ISOTHERMAL, NOSLIP, OUTFLOW, WALL, _channel_builder

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2511_17551_gb300 as dg
    dg.lib()
    return dg


RUNS = [("box", 3, 3, (1, 1, 1), NS), ("box", 3, 3, (20, 17, 9), NS), ("box", 3, 4, (12, 10, 9), NS), ("box", 3, 7, (7, 5, 9), {}),
        ("box", 3, 7, (3, 2, 3), dict(alpha_max=0.5, positivity_eps=0.1, **NS)),
        ("box", 2, 3, (90, 61), dict(alpha_max=0.5, positivity_eps=0.1)),
        ("channel", 3, 3, (9, 8, 7), dict(bc_kind=[INFLOW, OUTFLOW], bc_prim=np.array([INFLOW_STATE] * 2), **NS)),
        ("channel", 3, 4, (3, 8, 7), dict(bc_kind=[NOSLIP, ISOTHERMAL], bc_prim=np.array([WALL] * 2), **NS)),
        ("mixture", 3, 4, (6, 8, 5), {}), ("mixture", 3, 3, (2, 4, 1), {}), ("chemistry", 3, 4, (6, 8, 5), {})]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kind,dim,N,shape,kw", RUNS)
def test_overlapped_launches_change_nothing(dg, precision, kind, dim, N, shape, kw):
    kw = dict(kw)
    if kind in ("mixture", "chemistry"):
        build = _mixture(shape)
        kinds, bcp = cases.mixture_bc(cases.mixture_ogrid(dg.dg_lgl_nodes(N)[0], *shape)[3])
        kw = dict(n_species=5, species=W.species_table(), volume_flux=1, bc_kind=kinds, bc_prim=bcp, alpha_max=0.5,
                  positivity_eps=0.1)
        if kind == "chemistry":
            kw["reactions"] = W.reaction_table()
    else:
        build = _box(shape, dim) if kind == "box" else _channel_builder(shape)
    xyz, nbr, face, w = build(dg.dg_lgl_nodes(N)[0])
    s = dg.Solver(dim, N, xyz, nbr, face, precision=precision, **kw)
    try:
        if kind == "channel":
            w = cases.perturbed_state(w, 5, amp=0.05)
        got = []
        for apart in (1, 0, 0):
            dg.dg_profile(s.ctx, apart)
            s.set_primitive(w)
            # (chemistry from a perturbed cold flow stays physical at a twentieth)
            t = s.step(4, cfl=0.01 if kind == "chemistry" else 0.2)
            u, _ = s.get_state()
            got.append((t, np.array(u)))
        for t, u in got[1:]:
            assert t == got[0][0] and np.array_equal(u, got[0][1])
        assert np.all(np.isfinite(got[0][1]))
    finally:
        s.close()


@pytest.mark.parametrize("batch,n_out,own_stream", [(1, 1, False), (200, 10, True), (4096, 10, False), (5000, 1, True)])
def test_overlapped_training_changes_nothing(dg, batch, n_out, own_stream):
    """Training iterations (two gathers into buffers that the last iteration read, gradient, Adam) with a
    synchronisation after each call and without any."""
    import torch
    g = torch.Generator().manual_seed(3)
    X = torch.randn((20000, 7), generator=g).cuda()
    Y = torch.randn((20000, n_out), generator=g).cuda()
    idx = torch.randint(0, 20000, (30, batch), generator=g).cuda()
    P0 = (0.3 * torch.randn((dg.dg_mlp_nparams(n_out),), generator=g)).cuda()
    stream = torch.cuda.Stream() if own_stream else None
    raw = stream.cuda_stream if own_stream else None
    got = []
    for apart in (True, False, False):
        P, m, v = P0.clone(), torch.zeros_like(P0), torch.zeros_like(P0)
        loss = torch.zeros((1,), dtype=torch.float64, device="cuda")
        ws = torch.empty((dg.dg_mlp_workspace_bytes(batch, n_out) // 4,), device="cuda")
        xb, yb = torch.empty((batch, 7), device="cuda"), torch.empty((batch, n_out), device="cuda")
        torch.cuda.synchronize()
        wait = torch.cuda.synchronize if apart else (lambda: None)
        for k in range(30):
            dg.dg_gather_rows(X, idx[k], xb, raw), wait()
            dg.dg_gather_rows(Y, idx[k], yb, raw), wait()
            dg.dg_mlp_train_step(P, m, v, xb, yb if n_out > 1 else yb.reshape(-1), k + 1, 1e-3, loss, ws, raw), wait()
        torch.cuda.synchronize()
        got.append((P, m, v, loss))
    for other in got[1:]:
        assert all(torch.equal(a, b) for a, b in zip(got[0], other))
    assert torch.isfinite(got[0][0]).all() and not torch.equal(got[0][0], P0)


def _reacting(dg, precision, stream=None):
    x, _ = dg.dg_lgl_nodes(4)
    xyz, nbr, face, w = cases.mixture_ogrid(x, 6, 8, 5, hot=(1.2, 2500.0))
    kinds, bcp = cases.mixture_bc(w)
    s = dg.Solver(3, 4, xyz, nbr, face, n_species=5, species=W.species_table(), volume_flux=1, bc_kind=kinds, bc_prim=bcp,
                  alpha_max=0.5, precision=precision, reactions=W.reaction_table(), stream=stream)
    s.set_primitive(w)
    return s


def _learn(dg, s, which):
    """A network that is far off: the source's box ends at 1200 K, so that some tiles are accepted (the floor is
    wide) and others recomputed; the temperature's is corrected by Newton steps."""
    rng = np.random.default_rng(3)
    if which == dg.DG_SURROGATE_TEMPERATURE:
        p = (0.1 * rng.normal(size=dg.dg_mlp_nparams(1))).astype(np.float32)
        st = np.concatenate([np.zeros(7), np.ones(7), [600.0, 200.0]])
        st[13], st[12] = 1e6, 5.0
    else:
        p = (0.1 * rng.normal(size=dg.dg_mlp_nparams(10))).astype(np.float32)
        st = np.zeros(53)
        st[7:14], st[24:34], st[34], st[35] = [1, 1, 1, 1, 1, 5, 1000], 1.0, 1e-3, 1.0
        st[36:43], st[43:50], st[50:53] = -1e30, 1e30, [0.1, 1e30, 1.0]
        st[49] = 1200.0
    dg.dg_set_surrogate(s.ctx, p, st, which=which)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("which,refresh", [("source", 0), ("source", 1), ("source", 2), ("temperature", 0)])
def test_overlapped_learned_launches_change_nothing(dg, precision, which, refresh):
    """The learned source (its tile counter, sampled checks, fallback and corrections) and the learned
    temperature in steps, kept apart and overlapped: the same bits and the same decisions."""
    got = []
    for apart in (1, 0, 0):
        s = _reacting(dg, precision)
        try:
            k = dg.DG_SURROGATE_SOURCE if which == "source" else dg.DG_SURROGATE_TEMPERATURE
            _learn(dg, s, k)
            if refresh:
                dg.dg_set_source_refresh(s.ctx, refresh)
            dg.dg_profile(s.ctx, apart)
            t = s.step(4, cfl=0.01)
            got.append((t, np.array(s.get_state()[0]), dg.dg_surrogate_stats(s.ctx, k), dg.dg_get_source(s.ctx, s.shape)[:2]))
        finally:
            s.close()
    accepted, recomputed = got[0][2]
    print(which, refresh, "accepted, recomputed", accepted, recomputed)
    assert recomputed > 0 and (which == "temperature" or accepted > 0)
    for t, u, n, (S, flags) in got[1:]:
        assert t == got[0][0] and n == got[0][2] and np.array_equal(u, got[0][1])
        assert np.array_equal(S, got[0][3][0]) and np.array_equal(flags, got[0][3][1])


def _edges(raw, call):
    """(edges, programmatic ones) of the graph that `call` makes on the stream `raw`; nothing runs."""
    import ctypes as C
    rt = C.CDLL("libcudart.so.13")
    graph, n = C.c_void_p(), C.c_size_t(0)
    assert rt.cudaStreamBeginCapture(C.c_void_p(raw), 2) == 0
    try:
        call()
    finally:
        assert rt.cudaStreamEndCapture(C.c_void_p(raw), C.byref(graph)) == 0
    assert rt.cudaGraphGetEdges(graph, None, None, None, C.byref(n)) == 0
    a, b = (C.c_void_p * n.value)(), (C.c_void_p * n.value)()
    data = (C.c_uint8 * (8 * n.value))()  # cudaGraphEdgeData: two ports, the type (1: programmatic), reserved
    assert rt.cudaGraphGetEdges(graph, a, b, data, C.byref(n)) == 0
    assert rt.cudaGraphDestroy(graph) == 0
    return n.value, sum(1 for i in range(n.value) if data[8 * i + 2] == 1)


@pytest.mark.parametrize("kind", ["channel", "learned"])
def test_timed_kernels_are_launched_apart(dg, kind):
    """The reference arm of this file: while kernels are timed none is launched to overlap, nor within the
    chains that share one pair of events (gradients and boundary lifting, the learned source's kernels)."""
    import torch
    stream = torch.cuda.Stream()
    if kind == "learned":
        s = _reacting(dg, 1, stream.cuda_stream)
        _learn(dg, s, dg.DG_SURROGATE_SOURCE)
    else:
        x, _ = dg.dg_lgl_nodes(3)
        xyz, nbr, face, w = _channel_builder((3, 4, 3))(x)
        s = dg.Solver(3, 3, xyz, nbr, face, precision=1, bc_kind=[NOSLIP, ISOTHERMAL], bc_prim=np.array([WALL] * 2),
                      stream=stream.cuda_stream, **NS)
        s.set_primitive(w)
    try:
        u = torch.from_numpy(s.get_state()[0]).cuda().float()
        r = torch.empty_like(u)
        dg.dg_rhs(s.ctx, u, r)
        dg.dg_sync(s.ctx)
        n, overlapped = _edges(stream.cuda_stream, lambda: dg.dg_rhs(s.ctx, u, r))
        assert n >= 2 and overlapped >= 2, (n, overlapped)
        dg.dg_profile(s.ctx, 1)
        assert _edges(stream.cuda_stream, lambda: dg.dg_rhs(s.ctx, u, r)) == (n, 0)
    finally:
        s.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_rhs_between_the_callers_kernels(dg, precision):
    """dg_rhs on the caller's stream between kernels that write its input and read its output."""
    import torch
    stream = torch.cuda.Stream()
    xyz, nbr, face, w = _box((20, 17, 9), 3)(dg.dg_lgl_nodes(3)[0])
    s = dg.Solver(3, 3, xyz, nbr, face, precision=precision, stream=stream.cuda_stream, **NS)
    try:
        s.set_primitive(w)
        u0 = torch.from_numpy(s.get_state()[0]).cuda()
        u0 = u0.float() if precision else u0
        got = []
        for apart in (True, False, False):
            u, r, total = u0.clone(), torch.empty_like(u0), torch.zeros_like(u0)
            torch.cuda.synchronize()
            wait = torch.cuda.synchronize if apart else (lambda: None)
            with torch.cuda.stream(stream):
                for k in range(12):
                    u.mul_(1.0 + 1e-3 * k), wait()
                    dg.dg_rhs(s.ctx, u, r), wait()
                    total.add_(r), wait()
                    r.fill_(float("nan")), wait()
            torch.cuda.synchronize()
            got.append(total)
        assert torch.isfinite(got[0]).all() and all(torch.equal(got[0], g) for g in got[1:])
    finally:
        s.close()


@pytest.mark.parametrize("N,n_el", [(3, 4), (4, 4), (4, 6)])
def test_captured_allocation_free_rhs(dg, N, n_el):
    """dg_rhs_ns_noalloc in a CUDA graph, between kernels that write its metric terms and input and read its
    output, replayed on new values: the bits of a plain call."""
    import torch
    x, _ = dg.dg_lgl_nodes(N)
    xyz, nbr, face, w = cases.tgv(x, n_el, warp=0.1)
    s = dg.Solver(3, N, xyz, nbr, face, equations=dg.DG_NAVIER_STOKES, mu=0.01, Pr=0.72)
    try:
        s.set_primitive(cases.perturbed_state(w, 1))
        u0 = torch.from_numpy(s.get_state()[0]).cuda()
        Ja0 = torch.empty((s.K, 3, 3, s.np), dtype=torch.float64, device="cuda")
        iJ0 = torch.empty((s.K, s.np), dtype=torch.float64, device="cuda")
        dg.dg_get_metrics(s.ctx, Ja0, iJ0)
        nb = torch.from_numpy(np.ascontiguousarray(nbr, dtype=np.int32)).cuda()
        scale = torch.ones((), dtype=torch.float64, device="cuda")
        u, Ja, iJ, r, out = torch.empty_like(u0), torch.empty_like(Ja0), torch.empty_like(iJ0), torch.empty_like(u0), torch.empty_like(u0)

        def call(raw):
            dg.dg_rhs_ns_noalloc(N, s.K, nb, Ja, iJ, 1.4, 0.01, 0.72, 0, 0, u, r, raw)

        def chain():
            torch.mul(u0, scale, out=u)
            torch.mul(Ja0, scale, out=Ja)
            torch.mul(iJ0, scale, out=iJ)
            call(torch.cuda.current_stream().cuda_stream)
            torch.mul(r, 2.0, out=out)

        chain()  # the first call sets up the scratch
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            chain()
        for f in (1.0, 1.25, 0.75):
            scale.fill_(f)
            for t in (u, Ja, iJ, r, out):
                t.fill_(float("nan"))
            torch.cuda.synchronize()
            graph.replay()
            torch.cuda.synchronize()
            got = out.clone()
            for g in (lambda: torch.mul(u0, scale, out=u), lambda: torch.mul(Ja0, scale, out=Ja), lambda: torch.mul(iJ0, scale, out=iJ)):
                g()
            torch.cuda.synchronize()
            call(None)
            torch.cuda.synchronize()
            assert dg.dg_noalloc_status()[0] == dg.DG_OK
            assert torch.isfinite(got).all() and torch.equal(got, 2.0 * r)
    finally:
        s.close()
