"""EBB_REDUCE_AUTO in FP64 (three threads per tet below 8,192 tets, one thread
per tet from there on) and the zeroing that the maps overlap: every map, both
models, on either side of the limit and at ragged tet counts, against the
oracle; outputs that start unaligned and full of garbage are zeroed whole."""
import numpy as np
import pytest
import torch

import meshgen
from _problems import oracle_maps, problem, rel_err

pytestmark = pytest.mark.gpu


def _mesh(m, mu, lam):
    from paper_1506_07577_gb300.device_mesh import DeviceTetMesh
    return DeviceTetMesh(m.X, m.tets, mu, lam)


def _maps(dm, model, prec):
    from paper_1506_07577_gb300 import abi
    o = abi.map_opts(abi.EBB_STVK if model == "stvk" else abi.EBB_NEOHOOKEAN, precision=prec,
                     flags=abi.EBB_MAP_ZERO_OUT)
    abi.ebb_map_tet_force_Kv(dm.ctx, dm.tets, "u", "w", "f", "k", o)
    abi.ebb_map_tet_forces(dm.ctx, dm.tets, "u", "f2", o)
    abi.ebb_map_tet_Kv(dm.ctx, dm.tets, "u", "w", "k2", o)
    abi.ebb_map_tet_diagK(dm.ctx, dm.tets, "u", "d", o)
    abi.ebb_ctx_sync(dm.ctx)


# 40, 5,000 and 8,640 tets
@pytest.mark.parametrize("model", ["stvk", "nh"])
@pytest.mark.parametrize("n", [2, 10, 12])
def test_auto_f64_matches_oracle(model, n):
    from paper_1506_07577_gb300 import abi
    m, mu, lam, u, w = problem(n, model, seed=81, permute=True)
    f, kw, d = oracle_maps(m, mu, lam, u, w, model)
    with _mesh(m, mu, lam) as dm:
        dm.vertex_field("u", torch.float64, value=u)
        dm.vertex_field("w", torch.float64, value=w)
        out = {k: dm.vertex_field(k, torch.float64, value=np.full((m.n_verts, 3), np.nan))
               for k in ("f", "f2", "k", "k2", "d")}
        _maps(dm, model, abi.EBB_PREC_F64)
        got = {k: t.cpu().numpy().T for k, t in out.items()}
    for k, ref in (("f", f), ("f2", f), ("k", kw), ("k2", kw), ("d", d)):
        assert rel_err(got[k], ref) < 1e-12, k


# planes of 3 (n + 1)^3 floats that start 4, 8 and 12 bytes past a 16-byte bound
@pytest.mark.parametrize("shift", [1, 2, 3])
def test_zeroed_outputs_at_any_alignment(shift):
    from paper_1506_07577_gb300 import abi
    m, mu, lam, u, w = problem(3, "nh", seed=82)
    f, kw, d = oracle_maps(m, mu, lam, u, w, "nh")
    with _mesh(m, mu, lam) as dm:
        dm.vertex_field("u", torch.float32, value=u)
        dm.vertex_field("w", torch.float32, value=w)
        out = {}
        for k in ("f", "f2", "k", "k2", "d"):
            buf = torch.full((3 * m.n_verts + 8,), float("nan"), device=dm.device)
            out[k] = buf
            dm.bind(k, buf[shift:shift + 3 * m.n_verts].view(3, m.n_verts))
        _maps(dm, "nh", abi.EBB_PREC_F32)
        n = 3 * m.n_verts
        for k, ref in (("f", f), ("f2", f), ("k", kw), ("k2", kw), ("d", d)):
            b = out[k].cpu().numpy()
            assert rel_err(b[shift:shift + n].reshape(3, -1).T, ref) < 1e-5, k
            assert np.isnan(b[:shift]).all() and np.isnan(b[shift + n:]).all(), k
