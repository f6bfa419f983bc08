"""FP64 steps on the row matrix with rtol = 0, which iterate until the residual
underflows (or max_iters is reached): no error, and the oracle's result."""
import numpy as np
import pytest
import torch

import meshgen
from oracle import fem, implicit
from _problems import rel_err

pytestmark = pytest.mark.gpu

RHO = 1000.0


def _step(m, u, v, dt, rho, gravity, rtol):
    from paper_1506_07577_gb300 import abi
    from paper_1506_07577_gb300.device_mesh import DeviceTetMesh
    mu, lam = (float(x) for x in meshgen.lame_from_young(1e5, 0.45))
    with DeviceTetMesh(m.X, m.tets) as dm:
        tu = dm.vertex_field("u", torch.float64, value=u)
        tv = dm.vertex_field("v", torch.float64, value=v)
        dm.bind("pinned", torch.from_numpy(m.pinned.astype(np.uint8)).to(dm.device))
        prm = abi.step_params(abi.EBB_STVK, dt, rho, mu, lam, gravity, abi.EBB_PREC_F64, max_iters=2000, rtol=rtol)
        rep = abi.ebb_cg_implicit_step(dm.ctx, dm.tets, "u", "v", "pinned", prm)
        return tu.cpu().numpy().T.copy(), tv.cpu().numpy().T.copy(), rep


def _oracle(m, u, v, dt, rho, gravity, rtol):
    mu, lam = (float(x) for x in meshgen.lame_from_young(1e5, 0.45))
    B, V = fem.rest_shape(m.X, m.tets)
    mass = fem.lumped_mass(V, m.tets, rho, m.n_verts)
    return implicit.implicit_step(m.X, u, v, m.tets, B, V, mass, mu, lam, fem.STVK, dt, np.array(gravity), m.pinned,
                                  2000, rtol)


# 1e-11: both solves run to rounding, 1e-15 of the residual; kappa of the scaled A is at
# most 650 here, so that is below 1e-12 of the solution, plus the rounding of K and f
@pytest.mark.parametrize("n,dt,rho", [(1, 1e-3, RHO), (4, 1e-3, RHO), (8, 1e-3, RHO), (8, 1e-4, RHO), (8, 1e-2, RHO),
                                      (8, 1e-3, 1e-5 * RHO), (14, 1e-3, RHO)])
def test_zero_tolerance(n, dt, rho):
    m = meshgen.cube_grid(n, jitter=0.01, seed=1)
    u = meshgen.random_displacement(m.X, n, amp=0.02, seed=2, smooth=0.01)
    v = 0.05 * meshgen.random_field(m.n_verts, seed=3)
    g = (0.0, 0.0, -9.81)
    ug, vg, rep = _step(m, u, v, dt, rho, g, 0.0)
    uo, vo, _ = _oracle(m, u, v, dt, rho, g, 1e-15)
    assert rep.status == 0 and rep.rel_residual < 1e-16
    assert rel_err(vg, vo) < 1e-11 and rel_err(ug, uo) < 1e-11
