"""FP64 implicit steps on the assembled row matrix, at the sizes where its
layout can go wrong: fewer vertices than one slice, window and slice edges,
both forms of the solve, long rows, and rows too long for it (the matrix-free
step then runs).  Compared with the FP64 oracle's step.

Tolerance: with CG run to rtol 1e-14 the two solves differ by about kappa(A)
times that; dt makes A mass-dominated (kappa below 100), so 1e-12 leaves room
for rounding only."""
import numpy as np
import pytest
import torch

import meshgen
from oracle import fem, implicit
from _problems import rel_err

pytestmark = pytest.mark.gpu

G = (0.0, 0.0, -9.81)
RHO = 1000.0


def _step(X, tets, mu, lam, model, u, v, pinned, dt, reps=2):
    """`reps` steps on the GPU and by the oracle; both final states."""
    from paper_1506_07577_gb300 import abi
    from paper_1506_07577_gb300.device_mesh import DeviceTetMesh
    per_tet = np.ndim(mu) > 0
    with DeviceTetMesh(X, tets, mu if per_tet else None, lam if per_tet else None) as dm:
        tu = dm.vertex_field("u", torch.float64, value=u)
        tv = dm.vertex_field("v", torch.float64, value=v)
        name = None
        if pinned is not None:
            name = "pinned"
            dm.bind(name, torch.from_numpy(pinned).to(dm.device))
        prm = abi.step_params(abi.EBB_STVK if model == "stvk" else abi.EBB_NEOHOOKEAN, dt, RHO,
                              0.0 if per_tet else mu, 0.0 if per_tet else lam, G, abi.EBB_PREC_F64,
                              max_iters=500, rtol=1e-14)
        for _ in range(reps):
            abi.ebb_cg_implicit_step(dm.ctx, dm.tets, "u", "v", name, prm)
        got = tu.cpu().numpy().T.copy(), tv.cpu().numpy().T.copy()
    B, V = fem.rest_shape(X, tets)
    mass = fem.lumped_mass(V, tets, RHO, X.shape[0])
    pin = np.zeros(X.shape[0], bool) if pinned is None else pinned != 0
    for _ in range(reps):
        u, v, _ = implicit.implicit_step(X, u, v, tets, B, V, mass, mu, lam,
                                         fem.STVK if model == "stvk" else fem.NEOHOOKEAN, dt, np.array(G), pin, 500,
                                         1e-14)
    return got, (u, v)


@pytest.mark.parametrize("model", ["stvk", "nh"])
# vertices: 8 (one slice), 27, 343 (past one window), 4,096 and 4,913 (either
# side of the limit between the two forms of the solve)
@pytest.mark.parametrize("n,pin", [(1, None), (2, "u8"), (6, "i32"), (15, "u8"), (16, "u8")])
def test_row_step_matches_oracle(model, n, pin):
    m = meshgen.cube_grid(n, jitter=0.02, seed=71 + n, permute=n == 6)
    mu, lam = (float(x) for x in meshgen.lame_from_young(1e5, 0.45)) if n == 15 else \
        meshgen.material_perturbed_lame(m.n_tets, 1e5, 0.4, 0.2, seed=n)
    u = meshgen.random_displacement(m.X, n, amp=0.02, seed=n, smooth=0.01)
    v = 0.05 * meshgen.random_field(m.n_verts, seed=n)
    pinned = None if pin is None else m.pinned.astype(np.uint8 if pin == "u8" else np.int32)
    (ug, vg), (uo, vo) = _step(m.X, m.tets, mu, lam, model, u, v, pinned, 1e-4)
    assert rel_err(vg, vo) < 1e-12 and rel_err(ug, uo) < 1e-12


# hub vertices in 96 tets (a long row) and in 384 (more than a row may have)
@pytest.mark.parametrize("segments,apexes", [(4, 24), (16, 24)])
def test_row_step_on_long_rows(segments, apexes):
    m = meshgen.hub_fan(segments, apexes, seed=72)
    mu, lam = (float(x) for x in meshgen.lame_from_young(1e5, 0.3))
    u = 0.01 * meshgen.random_field(m.n_verts, seed=1)
    v = 0.05 * meshgen.random_field(m.n_verts, seed=2)
    (ug, vg), (uo, vo) = _step(m.X, m.tets, mu, lam, "stvk", u, v, None, 1e-4)
    assert rel_err(vg, vo) < 1e-12 and rel_err(ug, uo) < 1e-12


def test_row_step_is_reproducible():
    from paper_1506_07577_gb300 import abi
    from paper_1506_07577_gb300.device_mesh import DeviceTetMesh
    m = meshgen.cube_grid(7, jitter=0.02, seed=73)
    mu, lam = (float(x) for x in meshgen.lame_from_young(1e5, 0.45))
    outs = []
    with DeviceTetMesh(m.X, m.tets) as dm:
        for _ in range(3):
            u = dm.vertex_field("u", torch.float64, value=meshgen.random_displacement(m.X, 7, amp=0.02, seed=3))
            v = dm.vertex_field("v", torch.float64)
            prm = abi.step_params(abi.EBB_STVK, 1e-3, RHO, mu, lam, G, abi.EBB_PREC_F64, rtol=1e-10)
            abi.ebb_cg_implicit_step(dm.ctx, dm.tets, "u", "v", None, prm)
            outs.append(torch.stack([u, v]).cpu().numpy())
    assert np.array_equal(outs[0], outs[1]) and np.array_equal(outs[0], outs[2])
