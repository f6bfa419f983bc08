"""FP32 batched steps solved in one launch per group of meshes: batches whose
border between the groups falls inside a tile, meshes smaller than a block's
share of vertices, one mesh, unequal meshes, a mesh without tets, and more
meshes than the one-launch form takes.  Every mesh is compared with the oracle's
step of that mesh alone (1e-5: FP32 element arithmetic, as in the batched tests)."""
import numpy as np
import pytest
import torch

import meshgen
from oracle import fem, implicit
from _problems import rel_err

pytestmark = pytest.mark.gpu

G = np.array([0.0, 0.0, -9.81])


def _run(b, model, u, v, X=None, batch=None, pinned=None):
    from paper_1506_07577_gb300 import abi
    from paper_1506_07577_gb300.device_mesh import DeviceTetMesh
    X = b.X if X is None else X
    batch = b.batch if batch is None else batch
    pinned = b.pinned if pinned is None else pinned
    mu, lam = (float(x) for x in meshgen.lame_from_young(1e5, 0.4))
    with DeviceTetMesh(X, b.tets, batch=batch) as dm:
        tu = dm.vertex_field("u", torch.float64, value=u)
        tv = dm.vertex_field("v", torch.float64, value=v)
        dm.bind("pinned", torch.from_numpy(pinned.astype(np.uint8)).to(dm.device))
        prm = abi.step_params(abi.EBB_STVK if model == "stvk" else abi.EBB_NEOHOOKEAN, 1e-3, 1000.0, mu, lam, tuple(G),
                              abi.EBB_PREC_F32, rtol=1e-8)
        reps = abi.ebb_cg_implicit_step_batched(dm.ctx, dm.tets, "u", "v", "pinned", "batch", int(batch[-1]) + 1, prm)
        return tu.cpu().numpy().T.copy(), tv.cpu().numpy().T.copy(), reps, mu, lam


@pytest.mark.parametrize("model", ["stvk", "nh"])
@pytest.mark.parametrize("sides", [[3], [2, 3], [3, 3, 3], [1, 6, 2, 5, 1, 4], [2] * 40])
def test_groups_match_oracle(model, sides):
    b = meshgen.cube_grid_batch(np.array(sides), jitter=0.02, seed=90)
    rng = np.random.default_rng(91)
    u = 0.002 * rng.normal(size=b.X.shape)
    v = 0.05 * rng.normal(size=b.X.shape)
    ug, vg, reps, mu, lam = _run(b, model, u, v)
    for m in range(len(sides)):
        X, tets, pin = b.mesh(m)
        s = slice(b.vert_off[m], b.vert_off[m + 1])
        B, V = fem.rest_shape(X, tets)
        mass = fem.lumped_mass(V, tets, 1000.0, X.shape[0])
        uo, vo, _ = implicit.implicit_step(X, u[s], v[s], tets, B, V, mass, mu, lam,
                                           fem.STVK if model == "stvk" else fem.NEOHOOKEAN, 1e-3, G, pin, 1000, 1e-8)
        assert reps[m].rel_residual <= 1e-8
        assert rel_err(vg[s], vo) < 1e-5 and rel_err(ug[s], uo) < 1e-5, m


# 2,500 meshes: more than 16 per SM, solved by the captured launches
def test_very_many_meshes_equal_one():
    b = meshgen.cube_grid_batch(np.full(2500, 1), jitter=0.0, seed=0)
    u = np.zeros_like(b.X)
    v = np.tile(0.05 * np.random.default_rng(3).normal(size=(8, 3)), (2500, 1))
    _, vg, reps, _, _ = _run(b, "stvk", u, v)
    per = vg.reshape(2500, 8, 3)
    assert rel_err(per, np.broadcast_to(per[:1], per.shape)) < 1e-5
    assert all(r.rel_residual <= 1e-8 for r in reps)


# a last mesh of pinned vertices without tets: the second group has no tiles
def test_group_without_tets():
    b = meshgen.cube_grid_batch(np.array([3]), jitter=0.02, seed=92)
    n = b.X.shape[0]
    X = np.concatenate([b.X, b.X + 2.0])
    batch = np.concatenate([np.zeros(n, np.int32), np.ones(n, np.int32)])
    pinned = np.concatenate([b.pinned, np.ones(n, bool)])
    rng = np.random.default_rng(93)
    u, v = 0.002 * rng.normal(size=X.shape), 0.05 * rng.normal(size=X.shape)
    ug, vg, reps, mu, lam = _run(b, "nh", u, v, X, batch, pinned)
    B, V = fem.rest_shape(b.X, b.tets)
    mass = fem.lumped_mass(V, b.tets, 1000.0, n)
    uo, vo, _ = implicit.implicit_step(b.X, u[:n], v[:n], b.tets, B, V, mass, mu, lam, fem.NEOHOOKEAN, 1e-3, G,
                                       b.pinned, 1000, 1e-8)
    assert rel_err(vg[:n], vo) < 1e-5 and rel_err(ug[:n], uo) < 1e-5
    assert np.array_equal(vg[n:], v[n:]) and reps[1].iters == 0
