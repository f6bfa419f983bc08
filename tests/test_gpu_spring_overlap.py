"""Overlapped spring steps read what the step before wrote: a run of many steps
(each launched while the last one ends) equals as many runs of one step (each
launch after the last one), bit for bit."""
import numpy as np
import pytest
import torch

import meshgen

pytestmark = pytest.mark.gpu


# 20^3: 9,261 rows, about one block per two SMs; 40^3: 68,921 rows, several waves
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("n,steps", [(20, 64), (40, 33)])
def test_run_equals_single_steps(dtype, n, steps):
    from paper_1506_07577_gb300 import abi
    from paper_1506_07577_gb300.device_mesh import DeviceTetMesh
    m = meshgen.cube_grid(n, jitter=0.05, seed=8)
    rng = np.random.default_rng(9)
    q0 = m.X + 0.01 * rng.normal(size=m.X.shape) / n
    qd0 = 0.2 * rng.normal(size=m.X.shape)
    mass = rng.uniform(0.5, 2.0, size=m.n_verts)
    out = []
    with DeviceTetMesh(m.X, m.tets, edges=True) as dm:
        dm.vertex_field("pos", dtype, value=m.X)
        abi.ebb_springs_init(dm.ctx, dm.tets, "pos")
        dm.vertex_field("mass", dtype, ncomp=1, value=mass)
        for runs, per_run in ((1, steps), (steps, 1)):
            q = dm.vertex_field("q", dtype, value=q0)
            qd = dm.vertex_field("qd", dtype, value=qd0)
            for _ in range(runs):
                abi.ebb_springs_run(dm.ctx, dm.tets, "q", "qd", "mass", 3.0, 1e-3, per_run)
                abi.ebb_ctx_sync(dm.ctx)
            out.append((q.clone(), qd.clone()))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert bool(torch.isfinite(out[0][0]).all())
