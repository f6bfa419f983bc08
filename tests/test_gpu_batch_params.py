"""Batched steps whose parameters change from call to call on one relation: each call
uses its own, as on a relation that saw no other.  In FP64 and in FP32 with another
reduction the CG iterations are recorded launches that keep their parameters."""
import numpy as np
import pytest
import torch

import meshgen

pytestmark = pytest.mark.gpu

G = (0.0, 0.0, -9.81)


def _mesh(b):
    from paper_1506_07577_gb300.device_mesh import DeviceTetMesh
    dm = DeviceTetMesh(b.X, b.tets, batch=b.batch)
    dm.vertex_field("u", torch.float64)
    dm.vertex_field("v", torch.float64)
    dm.bind("pinned", torch.from_numpy(b.pinned.astype(np.uint8)).to(dm.device))
    return dm


def _step(dm, b, prec, model, reduce, **change):
    from paper_1506_07577_gb300 import abi
    k = dict(mu=3e4, lam=5e4, rho=1000.0, dt=1e-3, rtol=1e-10, gravity=G)
    k.update(change)
    u, v = dm._tensors["u"], dm._tensors["v"]   # the same memory in every call
    u.copy_(torch.from_numpy(0.002 * meshgen.random_field(b.X.shape[0], seed=11).T))
    v.copy_(torch.from_numpy(0.05 * meshgen.random_field(b.X.shape[0], seed=12).T))
    torch.cuda.synchronize()
    prm = abi.step_params(abi.EBB_STVK if model == "stvk" else abi.EBB_NEOHOOKEAN, k["dt"], k["rho"], k["mu"],
                          k["lam"], k["gravity"], abi.EBB_PREC_F64 if prec == "f64" else abi.EBB_PREC_F32,
                          getattr(abi, "EBB_REDUCE_" + reduce), rtol=k["rtol"])
    abi.ebb_cg_implicit_step_batched(dm.ctx, dm.tets, "u", "v", "pinned", "batch", len(b.sides), prm)
    return u.clone(), v.clone()


@pytest.mark.parametrize("prec,reduce", [("f64", "AUTO"), ("f32", "ATOMIC"), ("f32", "TILED")])
def test_each_call_uses_its_parameters(prec, reduce):
    b = meshgen.cube_grid_batch(np.array([3, 5, 2]), jitter=0.02, seed=201)
    changes = [{}, {"lam": 2e5}, {"mu": 9e4}, {"mu": 9e4, "lam": 1e4}, {"dt": 2e-3}, {"rho": 500.0},
               {"gravity": (0.0, 5.0, 0.0)}, {}]
    # as many digits as the precisions' sums in any order have
    tol = 1e-9 if prec == "f64" else 1e-5
    for model in ("stvk", "nh"):
        with _mesh(b) as dm:
            got = [_step(dm, b, prec, model, reduce, **c) for c in changes]
        for c, g in zip(changes, got):
            with _mesh(b) as dm:
                want = _step(dm, b, prec, model, reduce, **c)
            for x, y in zip(g, want):
                assert float((x - y).abs().max()) <= tol * float(y.abs().max()), (model, c)


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_ids_changed_in_place_and_bound_again(prec):
    """Three grids as two meshes, first the first two together, then the last two, in
    the same memory.  Three CG iterations: their scalars are the meshes' own."""
    from paper_1506_07577_gb300 import abi
    b = meshgen.cube_grid_batch(np.array([4, 3, 4]), jitter=0.02, seed=202)
    splits = [np.array(s, np.int32)[b.batch] for s in ((0, 0, 1), (0, 1, 1))]
    prm = abi.step_params(abi.EBB_STVK, 5e-3, 1000.0, 3e4, 5e4, G,
                          abi.EBB_PREC_F64 if prec == "f64" else abi.EBB_PREC_F32, max_iters=3, rtol=1e-12)

    def run(dm, ids):
        dm._tensors["ids"].copy_(torch.from_numpy(ids))
        dm._tensors["u"].zero_()
        dm._tensors["v"].copy_(torch.from_numpy(0.05 * meshgen.random_field(b.X.shape[0], seed=13).T))
        torch.cuda.synchronize()
        dm.bind("ids", dm._tensors["ids"])
        abi.ebb_cg_implicit_step_batched(dm.ctx, dm.tets, "u", "v", "pinned", "ids", 2, prm)
        return dm._tensors["v"].clone()

    with _mesh(b) as dm:
        dm.vertex_field("ids", torch.int32, ncomp=1)
        got = [run(dm, splits[k]) for k in (0, 1, 0, 0)]
    want = []
    for k in (0, 1):
        with _mesh(b) as dm:
            dm.vertex_field("ids", torch.int32, ncomp=1)
            want.append(run(dm, splits[k]))
    tol = 1e-9 if prec == "f64" else 1e-5
    for g, k in zip(got, (0, 1, 0, 0)):
        assert float((g - want[k]).abs().max()) <= tol * float(want[k].abs().max())
    assert float((want[0] - want[1]).abs().max()) > 10 * tol * float(want[0].abs().max())
