"""Spring steps at the sizes where their slot layout can go wrong: fewer rows
than a warp, past one sorting window (1,024 rows) in a scattered numbering, and
rows of very unequal length; one step (which writes the caller's planes
directly) and odd and even counts of several."""
import numpy as np
import pytest
import torch

import meshgen
from oracle import springs
from _problems import rel_err

pytestmark = pytest.mark.gpu

# as in test_gpu_springs: FP64 rounding of sums of some 100 terms, FP32 element
# arithmetic over a few steps
TOL = {"f64": 1e-12, "f32": 1e-5}


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("steps", [1, 4, 5])
@pytest.mark.parametrize("mesh", ["one_cube", "scattered", "hub"])
def test_spring_slots_match_oracle(prec, steps, mesh):
    from paper_1506_07577_gb300 import abi
    from paper_1506_07577_gb300.device_mesh import DeviceTetMesh
    if mesh == "hub":
        m = meshgen.hub_fan(16, 24, seed=5)
    else:
        m = meshgen.cube_grid(1 if mesh == "one_cube" else 10, jitter=0.05, seed=6, permute=mesh == "scattered")
    rng = np.random.default_rng(7)
    q0 = m.X + 0.01 * rng.normal(size=m.X.shape)
    qd0 = 0.2 * rng.normal(size=m.X.shape)
    mass = rng.uniform(0.5, 2.0, size=m.n_verts)
    k, dt = 3.0, 1e-3
    dtype = torch.float64 if prec == "f64" else torch.float32
    with DeviceTetMesh(m.X, m.tets, edges=True) as dm:
        dm.vertex_field("pos", dtype, value=m.X)
        abi.ebb_springs_init(dm.ctx, dm.tets, "pos")
        q = dm.vertex_field("q", dtype, value=q0)
        qd = dm.vertex_field("qd", dtype, value=qd0)
        dm.vertex_field("mass", dtype, ncomp=1, value=mass)
        abi.ebb_springs_run(dm.ctx, dm.tets, "q", "qd", "mass", k, dt, steps)
        abi.ebb_ctx_sync(dm.ctx)
        got = q.double().cpu().numpy().T, qd.double().cpu().numpy().T
    e = springs.tet_edges(m.tets)
    want = springs.run(q0, qd0, mass, e, springs.rest_lengths(m.X, e), k, dt, steps)
    assert rel_err(got[0], want[0]) < TOL[prec] and rel_err(got[1], want[1]) < TOL[prec]
