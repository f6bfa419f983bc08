"""Assembled FP32 steps and products at tet counts around the blocks (64 tets) and
warps (32) of the element pass, on meshes with unused vertices, against the FP64
oracle.  A record written past the last would land in a neighbouring allocation:
the step's vectors and scalars lie next to them in some of these sizes."""
import numpy as np
import pytest
import torch

import meshgen
from oracle import fem, implicit
from _problems import rel_err

pytestmark = pytest.mark.gpu

G = (0.0, 0.0, -9.81)


@pytest.mark.parametrize("model", ["stvk", "nh"])
@pytest.mark.parametrize("nt", [1, 31, 32, 33, 63, 64, 65, 96, 97, 128, 129, 155, 157, 159, 160, 161, 192, 193])
def test_assembled_step_and_product(model, nt):
    from paper_1506_07577_gb300 import abi
    from paper_1506_07577_gb300.device_mesh import DeviceTetMesh
    m = meshgen.cube_grid(4, jitter=0.02, seed=211)
    rng = np.random.default_rng(nt)
    X = np.concatenate([m.X, rng.random((20, 3))])
    tets = m.tets[rng.permutation(m.n_tets)[:nt]]
    pin = np.ones(X.shape[0], bool)
    pin[np.unique(tets)] = False   # unused vertices have no mass
    pin |= rng.random(X.shape[0]) < 0.1
    mu, lam = (float(x) for x in meshgen.lame_from_young(1e5, 0.4))
    mdl = abi.EBB_STVK if model == "stvk" else abi.EBB_NEOHOOKEAN
    om = fem.STVK if model == "stvk" else fem.NEOHOOKEAN
    u, v, w = 0.002 * rng.normal(size=X.shape), 0.05 * rng.normal(size=X.shape), rng.normal(size=X.shape)
    B, V = fem.rest_shape(X, tets)
    mass = fem.lumped_mass(V, tets, 1000.0, X.shape[0])
    uo, vo, _ = implicit.implicit_step(X, u, v, tets, B, V, mass, mu, lam, om, 1e-3, np.array(G), pin, 500, 1e-12)
    Kw = fem.tet_Kv(X + u, w, tets, B, V, mu, lam, om, X.shape[0])
    with DeviceTetMesh(X, tets, edges=True) as dm:
        dm.bind("pinned", torch.from_numpy(pin.astype(np.uint8)).to(dm.device))
        for prec, dt, tol in ((abi.EBB_PREC_F64, torch.float64, 1e-9), (abi.EBB_PREC_F32, torch.float32, 1e-5)):
            dm.vertex_field("u", dt, value=u)
            dm.vertex_field("w", dt, value=w)
            kw = dm.vertex_field("kw", dt)
            o = abi.map_opts(mdl, mu, lam, prec, flags=abi.EBB_MAP_ZERO_OUT)
            abi.ebb_assemble_tet_K(dm.ctx, dm.tets, "u", o)
            abi.ebb_spmv_tet_K(dm.ctx, dm.tets, "w", "kw", o)
            abi.ebb_ctx_sync(dm.ctx)
            assert rel_err(kw.cpu().numpy().T, Kw) < tol
            su = dm.vertex_field("su", torch.float64, value=u)
            sv = dm.vertex_field("sv", torch.float64, value=v)
            prm = abi.step_params(mdl, 1e-3, 1000.0, mu, lam, G, prec, rtol=1e-11 if prec == abi.EBB_PREC_F64 else 1e-8,
                                  flags=abi.EBB_STEP_ASSEMBLED)
            rep = abi.ebb_cg_implicit_step(dm.ctx, dm.tets, "su", "sv", "pinned", prm)
            assert rep.status == abi.EBB_OK and 0 < rep.iters < 200
            assert rel_err(sv.cpu().numpy().T, vo) < tol and rel_err(su.cpu().numpy().T, uo) < tol
