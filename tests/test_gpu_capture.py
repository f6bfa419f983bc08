"""Calls under capture of the context's stream.  Asynchronous calls (maps, spring
runs) are recorded and give on replay what the plain call gives; calls that read
results back (steps) are refused, and leave nothing behind that a later call
would take for its own."""
import numpy as np
import pytest
import torch

import meshgen

pytestmark = pytest.mark.gpu

G = (0.0, 0.0, -9.81)


class _Capture:
    """Capture of stream `s`, whatever the captured call does to it."""

    def __init__(self, s):
        self.s, self.g = s, torch.cuda.CUDAGraph()

    def __enter__(self):
        self.ctx = torch.cuda.stream(self.s)
        self.ctx.__enter__()
        self.g.capture_begin(capture_error_mode="thread_local")
        return self.g

    def __exit__(self, *exc):
        try:
            self.g.capture_end()
        except RuntimeError:
            pass
        self.ctx.__exit__(None, None, None)
        torch.cuda.synchronize()


def _mesh(n=5, **kw):
    from paper_1506_07577_gb300.device_mesh import DeviceTetMesh
    s = torch.cuda.Stream()
    m = meshgen.cube_grid(n, jitter=0.02, seed=31)
    return m, s, DeviceTetMesh(m.X, m.tets, stream=s, **kw)


def _params(kind, rho):
    from paper_1506_07577_gb300 import abi
    mu, lam = (float(x) for x in meshgen.lame_from_young(1e5, 0.4))
    prec = abi.EBB_PREC_F64 if kind in ("f64", "vjp") else abi.EBB_PREC_F32
    return abi.step_params(abi.EBB_STVK, 1e-3, rho, mu, lam, G, prec, rtol=1e-10)


def _step(dm, m, kind, rho):
    """One step (or VJP) from the same start; the two fields it updates."""
    from paper_1506_07577_gb300 import abi
    a = dm.vertex_field("a", torch.float64, value=meshgen.random_displacement(m.X, 5, amp=0.02, seed=3, smooth=0.01))
    b = dm.vertex_field("b", torch.float64, value=0.05 * meshgen.random_field(m.n_verts, seed=4))
    if kind == "vjp":
        for k, name in enumerate(("u", "v")):
            dm.vertex_field(name, torch.float64, value=0.01 * meshgen.random_field(m.n_verts, seed=5 + k))
    dm.vertex_field("ids", torch.int32, ncomp=1, value=np.zeros(m.n_verts, np.int32))
    return (a, b), {
        "f64": lambda: abi.ebb_cg_implicit_step(dm.ctx, dm.tets, "a", "b", None, _params(kind, rho)),
        "f32": lambda: abi.ebb_cg_implicit_step(dm.ctx, dm.tets, "a", "b", None, _params(kind, rho)),
        "batched": lambda: abi.ebb_cg_implicit_step_batched(dm.ctx, dm.tets, "a", "b", None, "ids", 1,
                                                            _params(kind, rho)),
        "vjp": lambda: abi.ebb_cg_implicit_step_vjp(dm.ctx, dm.tets, "u", "v", None, "a", "b", None, None,
                                                    _params(kind, rho)),
    }[kind]


@pytest.mark.parametrize("kind", ["f64", "f32", "batched", "vjp"])
@pytest.mark.parametrize("used_before", [False, True])
def test_refused_step_leaves_nothing_behind(kind, used_before):
    """A step with another density, refused under capture, then called again
    outside: as on a relation that never saw the first call.  FP64 steps repeat bit
    for bit; FP32 ones to the rounding of their atomic sums."""
    from paper_1506_07577_gb300 import abi
    m, s, dm = _mesh()
    with dm:
        if used_before:
            _step(dm, m, kind, 1000.0)[1]()
        _, call = _step(dm, m, kind, 500.0)
        with _Capture(s):
            with pytest.raises(abi.EbbError) as ei:
                call()
        assert ei.value.status == abi.EBB_ERR_CUDA
        got, call = _step(dm, m, kind, 500.0)
        call()
    m, s, fresh = _mesh()
    with fresh:
        want, call = _step(fresh, m, kind, 500.0)
        call()
    for x, y in zip(got, want):
        if kind in ("f64", "vjp"):
            tol = 0.0 if kind == "f64" else 1e-12
        else:
            tol = 1e-5
        assert float((x - y).abs().max()) <= tol * float(y.abs().max())


def test_call_after_a_refused_first_use():
    """A first spring run allocates, which a capture refuses; the next run outside
    is not told of that error."""
    from paper_1506_07577_gb300 import abi
    m, s, dm = _mesh(edges=True)
    with dm:
        dm.vertex_field("pos", torch.float64, value=m.X)
        abi.ebb_springs_init(dm.ctx, dm.tets, "pos")
        abi.ebb_ctx_sync(dm.ctx)
        dm.vertex_field("mass", torch.float64, ncomp=1, value=np.ones(m.n_verts))
        dm.vertex_field("q", torch.float64, value=1.01 * m.X)
        dm.vertex_field("qd", torch.float64)
        torch.cuda.synchronize()
        with _Capture(s):
            with pytest.raises(abi.EbbError) as ei:
                abi.ebb_springs_run(dm.ctx, dm.tets, "q", "qd", "mass", 3.0, 1e-3, 2)
        assert ei.value.status == abi.EBB_ERR_CUDA
        abi.ebb_springs_run(dm.ctx, dm.tets, "q", "qd", "mass", 3.0, 1e-3, 2)
        abi.ebb_ctx_sync(dm.ctx)


# maps that zero their outputs (a zeroing launch that the map overlaps), in the forms
# that are launched so, and the ones that are not
@pytest.mark.parametrize("prec,reduce", [("f64", "AUTO"), ("f64", "ATOMIC"), ("f64", "TILED"), ("f32", "TILED"),
                                         ("f32", "COOP"), ("f32", "TILED_ORDERED"), ("f32", "GATHER")])
def test_captured_zeroing_map_replays(prec, reduce):
    from paper_1506_07577_gb300 import abi
    m, s, dm = _mesh(n=9)
    dt = torch.float64 if prec == "f64" else torch.float32
    opts = abi.map_opts(abi.EBB_NEOHOOKEAN, 1e4, 4e4, abi.EBB_PREC_F64 if prec == "f64" else abi.EBB_PREC_F32,
                        getattr(abi, "EBB_REDUCE_" + reduce), abi.EBB_MAP_ZERO_OUT)
    with dm:
        u = dm.vertex_field("u", dt, value=meshgen.random_displacement(m.X, 9, amp=0.02, seed=3, smooth=0.01))
        w = dm.vertex_field("w", dt, value=meshgen.random_field(m.n_verts, seed=4))
        f, kw = dm.vertex_field("f", dt), dm.vertex_field("kw", dt)
        call = lambda: abi.ebb_map_tet_force_Kv(dm.ctx, dm.tets, "u", "w", "f", "kw", opts)
        call()   # (first uses allocate)
        abi.ebb_ctx_sync(dm.ctx)
        u0, w0 = u.clone(), w.clone()
        with _Capture(s) as g:
            call()
        for scale in (1.0, -0.5, 1.0):
            u.copy_(scale * u0)
            w.copy_(scale * w0)
            f.fill_(7.0)
            kw.fill_(7.0)
            torch.cuda.synchronize()
            g.replay()
            g.replay()
            torch.cuda.synchronize()
            got = f.clone(), kw.clone()
            call()
            abi.ebb_ctx_sync(dm.ctx)
            # the same sums, in the order of the atomics
            tol = 1e-13 if prec == "f64" else 1e-5
            for x, y in zip(got, (f, kw)):
                assert float((x - y).abs().max()) <= tol * float(y.abs().max())


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_captured_spring_run_replays(dtype):
    from paper_1506_07577_gb300 import abi
    m, s, dm = _mesh(n=9, edges=True)
    with dm:
        dm.vertex_field("pos", dtype, value=m.X)
        abi.ebb_springs_init(dm.ctx, dm.tets, "pos")
        dm.vertex_field("mass", dtype, ncomp=1, value=np.linspace(0.5, 2.0, m.n_verts))
        q, qd = dm.vertex_field("q", dtype, value=1.01 * m.X), dm.vertex_field("qd", dtype)
        q0 = q.clone()
        torch.cuda.synchronize()
        run = lambda: abi.ebb_springs_run(dm.ctx, dm.tets, "q", "qd", "mass", 3.0, 1e-3, 5)
        for _ in range(3):
            run()
        abi.ebb_ctx_sync(dm.ctx)
        want = q.clone(), qd.clone()
        with _Capture(s) as g:
            run()
        q.copy_(q0)
        qd.zero_()
        torch.cuda.synchronize()
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        assert torch.equal(q, want[0]) and torch.equal(qd, want[1])
