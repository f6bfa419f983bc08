"""Calls under capture of the context's stream.  What a capture refuses leaves
nothing behind that a later call would take for its own."""
import numpy as np
import pytest
import torch

import meshgen

pytestmark = pytest.mark.gpu


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
