"""The matrix-free FP64 step and step VJP, which run where the row matrix does not
apply: a mesh with a vertex in 192 tets beside an ordinary grid, every scatter
variant, against the FP64 oracle.

Tolerances as in test_gpu_rows (CG to 1e-14, kappa(A) below 100 at this dt: 1e-12)
and in test_gpu_adjoint (1e-8)."""
import numpy as np
import pytest
import torch

import meshgen
from oracle import adjoint, fem, implicit
from _problems import rel_err

pytestmark = pytest.mark.gpu

G = (0.0, 0.0, -9.81)
RHO = 1000.0


def _mesh():
    """4^3 grid and, apart from it, 192 tets around one vertex (more than a row takes, fewer
    than a colouring may need colours); a layer pinned."""
    c, h = meshgen.cube_grid(4, jitter=0.02, seed=81), meshgen.hub_fan(16, 12, seed=82)
    X = np.concatenate([c.X, h.X + 4.0])
    tets = np.concatenate([c.tets, h.tets + c.n_verts]).astype(np.int32)
    return X, tets, np.concatenate([c.pinned, np.zeros(h.n_verts, bool)])


def _state(X, seed):
    return 0.002 * meshgen.random_field(X.shape[0], seed=seed), 0.05 * meshgen.random_field(X.shape[0], seed=seed + 1)


@pytest.mark.parametrize("model", ["stvk", "nh"])
@pytest.mark.parametrize("reduce", ["ATOMIC", "COLOR", "TILED", "GATHER", "TILED_ORDERED", "COOP", "AUTO"])
def test_step_matches_oracle(model, reduce):
    from paper_1506_07577_gb300 import abi
    from paper_1506_07577_gb300.device_mesh import DeviceTetMesh
    X, tets, pin = _mesh()
    mu, lam = meshgen.material_perturbed_lame(tets.shape[0], 1e5, 0.4, 0.2, seed=83)
    u, v = _state(X, 84)
    with DeviceTetMesh(X, tets, mu, lam, colour=reduce == "COLOR") as dm:
        tu, tv = dm.vertex_field("u", torch.float64, value=u), dm.vertex_field("v", torch.float64, value=v)
        dm.bind("pinned", torch.from_numpy(pin.astype(np.uint8)).to(dm.device))
        prm = abi.step_params(abi.EBB_STVK if model == "stvk" else abi.EBB_NEOHOOKEAN, 1e-4, RHO, 0.0, 0.0, G,
                              abi.EBB_PREC_F64, getattr(abi, "EBB_REDUCE_" + reduce), max_iters=500, rtol=1e-14)
        for _ in range(2):
            abi.ebb_cg_implicit_step(dm.ctx, dm.tets, "u", "v", "pinned", prm)
        ug, vg = tu.cpu().numpy().T.copy(), tv.cpu().numpy().T.copy()
    B, V = fem.rest_shape(X, tets)
    mass = fem.lumped_mass(V, tets, RHO, X.shape[0])
    for _ in range(2):
        u, v, _ = implicit.implicit_step(X, u, v, tets, B, V, mass, mu, lam,
                                         fem.STVK if model == "stvk" else fem.NEOHOOKEAN, 1e-4, np.array(G), pin, 500,
                                         1e-14)
    assert rel_err(vg, v) < 1e-12 and rel_err(ug, u) < 1e-12


@pytest.mark.parametrize("reduce", ["AUTO", "TILED", "GATHER"])
@pytest.mark.parametrize("at", [False, True])
def test_vjp_matches_oracle_adjoint(at, reduce):
    """`at`: the caller hands in the step's new velocity."""
    from paper_1506_07577_gb300 import abi
    from paper_1506_07577_gb300.device_mesh import DeviceTetMesh
    X, tets, pin = _mesh()
    mu, lam = meshgen.material_perturbed_lame(tets.shape[0], 1e5, 0.4, 0.2, seed=85)
    u, v = _state(X, 86)
    u[pin] = v[pin] = 0.0
    rng = np.random.default_rng(87)
    gu_out, gv_out = rng.normal(size=u.shape), rng.normal(size=v.shape)
    dt = 1e-3
    B, V = fem.rest_shape(X, tets)
    mass = fem.lumped_mass(V, tets, RHO, X.shape[0])
    gu, gv, gmu, glam, _ = adjoint.step_vjp(X, u, v, tets, B, V, mass, mu, lam, dt, np.array(G), pin, gu_out, gv_out)
    prm = abi.step_params(abi.EBB_STVK, dt, RHO, 0.0, 0.0, G, abi.EBB_PREC_F64, getattr(abi, "EBB_REDUCE_" + reduce),
                          max_iters=2000, rtol=1e-14)
    with DeviceTetMesh(X, tets, mu, lam) as dm:
        dm.vertex_field("u", torch.float64, value=u)
        dm.vertex_field("v", torch.float64, value=v)
        dm.bind("pinned", torch.from_numpy(pin.astype(np.uint8)).to(dm.device))
        tgu, tgv = (dm.vertex_field(n, torch.float64, value=g) for n, g in (("gu", gu_out), ("gv", gv_out)))
        tgmu = dm.bind_tets("gmu", torch.zeros(tets.shape[0], dtype=torch.float64, device=dm.device))
        tglam = dm.bind_tets("glam", torch.zeros(tets.shape[0], dtype=torch.float64, device=dm.device))
        if at:
            _, v1, _ = implicit.implicit_step(X, u, v, tets, B, V, mass, mu, lam, fem.STVK, dt, np.array(G), pin, 2000,
                                              1e-14)
            dm.vertex_field("v1", torch.float64, value=v1)
            abi.ebb_cg_implicit_step_vjp_at(dm.ctx, dm.tets, "u", "v", "v1", "pinned", "gu", "gv", "gmu", "glam", prm)
        else:
            abi.ebb_cg_implicit_step_vjp(dm.ctx, dm.tets, "u", "v", "pinned", "gu", "gv", "gmu", "glam", prm)
        assert rel_err(tgu.cpu().numpy().T, gu) < 1e-8 and rel_err(tgv.cpu().numpy().T, gv) < 1e-8
        assert rel_err(tgmu.cpu().numpy(), gmu) < 1e-8 and rel_err(tglam.cpu().numpy(), glam) < 1e-8
