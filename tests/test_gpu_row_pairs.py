"""FP64 steps on the assembled rows where each block is summed once and stored in
both of its rows: pinned vertices scattered over the mesh (pairs with one, both
or no pinned row), another pinned field on the same relation, then none, so that
nothing of an earlier step stays in the matrix; mesh sides on either side of the
limit between the two forms of the solve (2,744 and 3,375 vertices).  Compared
with the FP64 oracle's steps.

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


@pytest.mark.parametrize("n", [3, 13, 14])
def test_pinned_fields_in_turn(n):
    from paper_1506_07577_gb300 import abi
    from paper_1506_07577_gb300.device_mesh import DeviceTetMesh
    m = meshgen.cube_grid(n, jitter=0.02, seed=40 + n)
    mu, lam = (float(x) for x in meshgen.lame_from_young(1e5, 0.4))
    u = meshgen.random_displacement(m.X, n, amp=0.02, seed=n, smooth=0.01)
    v = 0.05 * meshgen.random_field(m.n_verts, seed=n)
    rng = np.random.default_rng(n)
    pins = [rng.random(m.n_verts) < 0.3, rng.random(m.n_verts) < 0.3, np.zeros(m.n_verts, bool)]
    B, V = fem.rest_shape(m.X, m.tets)
    mass = fem.lumped_mass(V, m.tets, 1000.0, m.n_verts)
    prm = abi.step_params(abi.EBB_STVK, 1e-4, 1000.0, mu, lam, G, abi.EBB_PREC_F64, max_iters=500, rtol=1e-14)
    with DeviceTetMesh(m.X, m.tets) as dm:
        tu = dm.vertex_field("u", torch.float64, value=u)
        tv = dm.vertex_field("v", torch.float64, value=v)
        for i, pin in enumerate(pins):
            dm.bind("pin%d" % i, torch.from_numpy(pin.astype(np.uint8)).to(dm.device))
            abi.ebb_cg_implicit_step(dm.ctx, dm.tets, "u", "v", "pin%d" % i, prm)
            u, v, _ = implicit.implicit_step(m.X, u, v, m.tets, B, V, mass, mu, lam, fem.STVK, 1e-4, np.array(G), pin,
                                             500, 1e-14)
            assert rel_err(tv.cpu().numpy().T, v) < 1e-12 and rel_err(tu.cpu().numpy().T, u) < 1e-12, i
