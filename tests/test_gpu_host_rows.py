"""The host-buffer map on packed rows that the GPU reaches itself: one, two and six
chunks, row counts that end inside a row block, buffers off 16-byte bounds,
scattered vertices, and pageable buffers (which take the copying form); against
the device call on the same inputs, whose sums differ by the order of FP32
additions only (1e-6 of the largest entry)."""
import numpy as np
import pytest
import torch

from _problems import problem, rel_err

pytestmark = pytest.mark.gpu


def _pinned(n, shift):
    return torch.zeros(3 * n + 8, dtype=torch.float32).pin_memory()[shift:shift + 3 * n].view(n, 3)


# 320, 40,000, 640,000 and 2,560,000 tets: about 3, 320, 5,100 and 20,300 tiles
@pytest.mark.parametrize("n,shift,permute", [(4, 0, False), (20, 1, True), (20, 0, False), (50, 2, False),
                                             (80, 0, False)])
def test_host_rows_equal_device_call(n, shift, permute):
    from paper_1506_07577_gb300 import abi
    from paper_1506_07577_gb300.device_mesh import DeviceTetMesh
    m, mu, lam, u, w = problem(n, "stvk", seed=31, amp=0.05, per_tet=False, permute=permute)
    nv = m.n_verts
    with DeviceTetMesh(m.X, m.tets) as dm:
        for k in ("u", "w", "f", "k", "f2", "k2"):
            dm.vertex_field(k, x4=True)
        o = abi.map_opts(abi.EBB_STVK, mu, lam, abi.EBB_PREC_F32, flags=abi.EBB_MAP_ZERO_OUT | abi.EBB_MAP_HOST_XYZ)
        for pin in (True, False):
            bufs = [_pinned(nv, shift) if pin else torch.zeros((nv, 3)) for _ in range(4)]
            bufs[0].copy_(torch.from_numpy(u))
            bufs[1].copy_(torch.from_numpy(w))
            for _ in range(2):   # the plan is built by the first call
                abi.ebb_map_tet_force_Kv_host(dm.ctx, dm.tets, "u", "w", "f", "k", *bufs, o)
            abi.ebb_map_tet_force_Kv(dm.ctx, dm.tets, "u", "w", "f2", "k2", o)
            abi.ebb_ctx_sync(dm.ctx)
            for host, field, ref in ((bufs[2], "f", "f2"), (bufs[3], "k", "k2")):
                dev = dm._tensors[field][:, :3].cpu()
                assert torch.equal(host, dev)
                assert rel_err(dev.numpy(), dm._tensors[ref][:, :3].cpu().numpy()) < 1e-6
