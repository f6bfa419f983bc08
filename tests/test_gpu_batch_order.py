"""FP32 batched steps on relations whose tets are not in the order of the batch's
meshes: ids bound after finalize (the tets then lie in one Morton order over all
meshes, which share a box), ids under another name than the "batch" field of
finalize, and a finer grouping than that field.  Every mesh against the oracle's
step of that mesh alone (1e-5: FP32 element arithmetic, as in the batched tests)."""
import numpy as np
import pytest
import torch

import meshgen
from oracle import fem, implicit
from _problems import rel_err

pytestmark = pytest.mark.gpu

G = np.array([0.0, 0.0, -9.81])


def _setup(sides, seed):
    b = meshgen.cube_grid_batch(np.array(sides), jitter=0.02, seed=seed)
    rng = np.random.default_rng(seed + 1)
    return b, 0.002 * rng.normal(size=b.X.shape), 0.05 * rng.normal(size=b.X.shape)


def _step(dm, ids, nmesh, name, u, v, pinned, model, **kw):
    from paper_1506_07577_gb300 import abi
    mu, lam = (float(x) for x in meshgen.lame_from_young(1e5, 0.4))
    tu = dm.vertex_field("u", torch.float64, value=u)
    tv = dm.vertex_field("v", torch.float64, value=v)
    dm.bind("pinned", torch.from_numpy(pinned.astype(np.uint8)).to(dm.device))
    dm.vertex_field(name, torch.int32, ncomp=1, value=ids)
    prm = abi.step_params(abi.EBB_STVK if model == "stvk" else abi.EBB_NEOHOOKEAN, 1e-3, 1000.0, mu, lam, tuple(G),
                          abi.EBB_PREC_F32, **kw)
    reps = abi.ebb_cg_implicit_step_batched(dm.ctx, dm.tets, "u", "v", "pinned", name, nmesh, prm)
    return tu.cpu().numpy().T.copy(), tv.cpu().numpy().T.copy(), reps


# finalize_batch: the ids bound as "batch" before finalize (None: no field);
# name: the field that the call takes
@pytest.mark.parametrize("model", ["stvk", "nh"])
@pytest.mark.parametrize("sides,finalize_batch,name", [
    ([12, 12], None, "batch"),
    ([5, 9, 3, 7], None, "mesh_of"),
    ([6, 7, 6], (0, 0, 0), "mesh_of"),
    ([4, 6, 6, 4], (0, 1, 1, 2), "batch"),
    ([6, 6], (1, 0), "mesh_of"),
])
def test_any_tet_order_matches_oracle(model, sides, finalize_batch, name):
    from paper_1506_07577_gb300.device_mesh import DeviceTetMesh
    b, u, v = _setup(sides, 190)
    fb = None if finalize_batch is None else np.array(finalize_batch, np.int32)[b.batch]
    with DeviceTetMesh(b.X, b.tets, batch=fb) as dm:
        ug, vg, reps = _step(dm, b.batch, len(sides), name, u, v, b.pinned, model, rtol=1e-8)
    mu, lam = (float(x) for x in meshgen.lame_from_young(1e5, 0.4))
    for m in range(len(sides)):
        X, tets, pin = b.mesh(m)
        s = slice(b.vert_off[m], b.vert_off[m + 1])
        B, V = fem.rest_shape(X, tets)
        mass = fem.lumped_mass(V, tets, 1000.0, X.shape[0])
        uo, vo, _ = implicit.implicit_step(X, u[s], v[s], tets, B, V, mass, mu, lam,
                                           fem.STVK if model == "stvk" else fem.NEOHOOKEAN, 1e-3, G, pin, 1000, 1e-8)
        assert reps[m].rel_residual <= 1e-8
        assert rel_err(vg[s], vo) < 1e-5 and rel_err(ug[s], uo) < 1e-5, m


# Tets that join vertices of two meshes couple them in K p; the same few
# iterations by separate launches (atomic reduction) take every tet too.
def test_tets_that_join_meshes():
    from paper_1506_07577_gb300 import abi
    from paper_1506_07577_gb300.device_mesh import DeviceTetMesh
    m = meshgen.cube_grid(8, jitter=0.02, seed=193)
    rng = np.random.default_rng(194)
    u, v = 0.002 * rng.normal(size=m.X.shape), 0.05 * rng.normal(size=m.X.shape)
    ids = (np.arange(m.n_verts) * 2 // m.n_verts).astype(np.int32)
    out = []
    for reduce in (abi.EBB_REDUCE_TILED, abi.EBB_REDUCE_ATOMIC):
        with DeviceTetMesh(m.X, m.tets) as dm:
            out.append(_step(dm, ids, 2, "ids", u, v, m.pinned, "nh", reduce=reduce, max_iters=3, rtol=1e-12)[:2])
    assert rel_err(out[0][1], out[1][1]) < 1e-5 and rel_err(out[0][0], out[1][0]) < 1e-5
