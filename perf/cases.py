"""The measured workloads: what programs built on this library have it do.

Each case is one call (or one short sequence of calls) through the public
entry points -- ``DeviceTetMesh``, the ``abi`` functions and ``rollout`` -- on
a seeded box mesh of nx x ny x nz cubes, five tets per cube.  Meshes, fields
and materials are made on the GPU from the seed alone; the mesh, its finalized
relation and its bound fields are what a program holds before the call.

``exact`` gives the same results in plain float64 torch, without the library.
"""
from __future__ import annotations

import math

import torch

from paper_1506_07577_gb300 import abi
from paper_1506_07577_gb300.autograd import rollout
from paper_1506_07577_gb300.device_mesh import DeviceTetMesh

RHO, DT, GZ = 1000.0, 1e-3, -9.81
SPRING_K, SPRING_DT = 1.0, 1e-4
ASSEMBLED_ROW = 15          # blocks in a row of the assembled stiffness, about

# ---- the cases ---------------------------------------------------------------


def _box(kind, name, nx, ny, nz, **more):
    return {"name": name, "kind": kind, "nx": nx, "ny": ny, "nz": nz, **more}


def listed():
    return [
        # The smallest mesh in use: one FP64 map over 2,560 tets, as a program that drives its own
        # integrator calls it many times a second.  Launches and latency are all of it.
        _box("map", "map_f64_8", 8, 8, 8, model="stvk", precision="f64", ops="fused", material="uniform",
             reduce="auto", order="grid"),
        # The 64^3 neo-Hookean mesh with a material per tet, forces and K w for an explicit or matrix-free solver.
        _box("map", "map_f32_64_nh", 64, 64, 64, model="nh", precision="f32x4", ops="fused", material="per_tet",
             reduce="auto", order="grid"),
        # The large mesh: 10.5 million tets whose vertices and tets come in no useful order (as a mesher emits them).
        _box("map", "map_f32_128_random", 128, 128, 128, model="stvk", precision="f32x4", ops="fused",
             material="uniform", reduce="auto", order="random"),
        # Bitwise reproducible forces on an odd-sized mesh, fields as planes (column stores) of FP32.
        _box("map", "map_f32_ordered_ragged", 57, 41, 23, model="nh", precision="f32", ops="force",
             material="per_tet", reduce="ordered", order="grid"),
        # The FP64 stiffness product alone, the operator of a program's own Krylov solver.
        _box("map", "map_f64_kv_ragged", 45, 37, 40, model="nh", precision="f64", ops="kv", material="per_tet",
             reduce="auto", order="grid"),
        # One implicit FP64 step of the small mesh: the interactive, latency-bound use.
        _box("step", "step_f64_8", 8, 8, 8, model="stvk", precision="f64", material="uniform", rtol=1e-14,
             max_iters=50),
        # One implicit step of the 64^3 mesh in mixed precision: the production form of the simulation.
        _box("step", "step_mixed_64", 64, 64, 64, model="nh", precision="f32", material="per_tet", rtol=1e-8,
             max_iters=1000),
        # One implicit step of each of 256 unequal meshes: batched assets, or a learning environment's copies.
        {"name": "batch_mixed_256", "kind": "batch", "count": 256, "n_lo": 4, "n_hi": 24, "precision": "f32"},
        # A differentiable rollout and its gradient by state and material: parameter identification.
        _box("rollout", "rollout_32", 32, 32, 32, steps=20, every=5),
        # The assembled stiffness and one product with it, for solvers that want the matrix.
        _box("assembled", "assembled_f32_64", 64, 64, 64, model="nh", precision="f32x4", material="per_tet"),
        # An explicit spring-mass simulation on the mesh's edges, a hundred steps and the energy.
        _box("springs", "springs_f32_64", 64, 64, 64, precision="f32", steps=100),
        # The fused map on a program's own page-locked host arrays: two fields in, two fields out.
        _box("host", "host_f32_96", 96, 96, 96, model="stvk"),
    ]


def _dims(rng, lo, hi):
    """A box of about lo to hi cubes (spread over the logarithm), each side up to 2.5 times another's."""
    cubes = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    a, b = math.exp(rng.uniform(-0.45, 0.45)), math.exp(rng.uniform(-0.45, 0.45))
    s = cubes ** (1.0 / 3.0)
    nx, ny = max(1, round(s * a)), max(1, round(s * b))
    nz = max(1, min(int(hi // (nx * ny)), round(cubes / (nx * ny))))
    return {"nx": nx, "ny": ny, "nz": nz}


def draw(rng):
    kind = rng.choice(["map", "map", "map", "map", "step", "step", "step", "batch", "rollout", "assembled", "springs",
                       "host"])
    model, material = rng.choice(["stvk", "nh"]), rng.choice(["uniform", "per_tet"])
    if kind == "map":
        precision = rng.choice(["f32x4", "f32x4", "f32", "f64"])
        c = dict(_dims(rng, 64, 64 ** 3 if precision == "f64" else 120 ** 3), model=model, precision=precision,
                 ops=rng.choice(["fused", "fused", "kv", "force"]), material=material,
                 reduce=rng.choice(["auto", "auto", "auto", "ordered"]), order=rng.choice(["grid", "random"]))
    elif kind == "step":
        precision = rng.choice(["f32", "f64"])
        c = dict(_dims(rng, 216, 40 ** 3 if precision == "f64" else 64 ** 3), model=model, precision=precision,
                 material=material, rtol=1e-8 if precision == "f32" else 1e-12, max_iters=1000)
    elif kind == "batch":
        lo = rng.randint(3, 6)
        c = {"count": round(math.exp(rng.uniform(math.log(8), math.log(256)))), "n_lo": lo,
             "n_hi": rng.randint(lo + 4, 24), "precision": "f32"}
    elif kind == "rollout":
        steps = rng.randint(4, 16)
        c = dict(_dims(rng, 216, 28 ** 3), steps=steps, every=rng.randint(1, 5))
    elif kind == "assembled":
        c = dict(_dims(rng, 216, 60 ** 3), model=model, precision=rng.choice(["f32x4", "f64"]), material=material)
    elif kind == "springs":
        c = dict(_dims(rng, 216, 64 ** 3), precision=rng.choice(["f32", "f32", "f64"]), steps=rng.randint(20, 100))
    else:
        c = dict(_dims(rng, 24 ** 3, 96 ** 3), model=model)
    return {"kind": kind, **c}


# ---- inputs --------------------------------------------------------------------
# A cube's five tets as corner offsets (di, dj, dk), positively oriented; odd cubes are mirrored so that neighbours
# cut their shared face along the same diagonal.
_CORNERS = [
    [((1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 1)), ((0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1)),
     ((1, 1, 0), (0, 1, 0), (1, 0, 0), (1, 1, 1)), ((1, 0, 1), (0, 0, 1), (1, 1, 1), (1, 0, 0)),
     ((0, 1, 1), (1, 1, 1), (0, 0, 1), (0, 1, 0))],
    [((0, 0, 0), (1, 1, 0), (1, 0, 1), (0, 1, 1)), ((1, 0, 0), (0, 0, 0), (1, 1, 0), (1, 0, 1)),
     ((0, 1, 0), (1, 1, 0), (0, 0, 0), (0, 1, 1)), ((0, 0, 1), (1, 0, 1), (0, 1, 1), (0, 0, 0)),
     ((1, 1, 1), (0, 1, 1), (1, 0, 1), (1, 1, 0))],
]


def _oriented(t):
    e = [[t[a][c] - t[0][c] for c in range(3)] for a in (1, 2, 3)]
    det = (e[0][0] * (e[1][1] * e[2][2] - e[1][2] * e[2][1]) - e[0][1] * (e[1][0] * e[2][2] - e[1][2] * e[2][0])
           + e[0][2] * (e[1][0] * e[2][1] - e[1][1] * e[2][0]))
    return t if det > 0 else (t[0], t[1], t[3], t[2])


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _uniform(g, shape, lo, hi):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _mesh(g, nx, ny, nz, order="grid"):
    """Rest positions X (N_v, 3), keys (N_t, 4), pinned bottom layer, spacing h."""
    dev = "cuda"
    h = 1.0 / max(nx, ny, nz)
    k, j, i = torch.meshgrid(*(torch.arange(n + 1, device=dev) for n in (nz, ny, nx)), indexing="ij")
    X = torch.stack([i, j, k], -1).reshape(-1, 3).double() * h
    X = X + torch.randn(X.shape, generator=g, device=dev, dtype=torch.float64) * (0.01 * h)
    pinned = (k.reshape(-1) == 0).to(torch.uint8)
    ck, cj, ci = torch.meshgrid(*(torch.arange(n, device=dev) for n in (nz, ny, nx)), indexing="ij")
    base = (ci + (nx + 1) * (cj + (ny + 1) * ck)).reshape(-1, 1, 1)
    odd = ((ci + cj + ck) & 1).reshape(-1)
    off = torch.tensor([[[c[0] + (nx + 1) * (c[1] + (ny + 1) * c[2]) for c in _oriented(t)] for t in cube]
                        for cube in _CORNERS], device=dev)
    keys = (base + off[odd]).reshape(-1, 4)
    perm = None
    if order == "random":
        perm = torch.randperm(X.shape[0], generator=g, device=dev)
        keys = keys[torch.randperm(keys.shape[0], generator=g, device=dev)]
    elif order == "curve":
        # numbered along a space-filling curve, as programs that care for locality number their meshes
        code = torch.zeros_like(i.reshape(-1))
        for b in range(8):
            for c, x in enumerate((i, j, k)):
                code |= ((x.reshape(-1) >> b) & 1) << (3 * b + c)
        perm = torch.argsort(code)
    if perm is not None:
        inv = torch.empty_like(perm)
        inv[perm] = torch.arange(perm.numel(), device=dev)
        X, pinned, keys = X[perm], pinned[perm], inv[keys]
    return X.contiguous(), keys.to(torch.int32).contiguous(), pinned.contiguous(), h


def _lame(E, nu):
    return E / (2.0 * (1.0 + nu)), E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu))


def _material(g, material, model, nt):
    """(mu, lambda): two numbers, or one value per tet."""
    if material == "uniform":
        return _lame(1e5, 0.45)
    if model == "nh":   # Young's modulus over two decades
        return _lame(torch.exp(_uniform(g, (nt,), math.log(1e4), math.log(1e6))), 0.4)
    mu, lam = _lame(1e5, 0.45)
    return mu * _uniform(g, (nt,), 0.8, 1.2), lam * _uniform(g, (nt,), 0.8, 1.2)


def _displacement(g, X, h, amp):
    """A smooth bend and noise of amp * h, in the caller's vertex order."""
    a = _uniform(g, (3,), 0.5, 1.5)
    u = _uniform(g, X.shape, -amp * h, amp * h)
    bend = torch.stack([torch.sin(math.pi * a[0] * X[:, 2]) * X[:, 1], torch.sin(math.pi * a[1] * X[:, 0]) * X[:, 2],
                        torch.cos(math.pi * a[2] * X[:, 1]) * X[:, 0]], 1)
    return u + 0.01 * bend


def _sides(case):
    """Mesh sides of a batch: spread over the logarithm, the same for every seed."""
    c, lo, hi = case["count"], case["n_lo"], case["n_hi"]
    return [round(lo * (hi / lo) ** (((m * 157) % c + 0.5) / c)) for m in range(c)]


def _inputs(case, seed):
    """Everything made from the seed, as float64 tensors in the caller's order."""
    g = _generator(seed)
    kind = case["kind"]
    d = {"batch": None}
    if kind == "batch":
        Xs, Ks, Ps, Bs, off = [], [], [], [], 0
        for m, n in enumerate(_sides(case)):
            X, keys, pinned, _ = _mesh(g, n, n, n)
            Xs.append(X)
            Ks.append(keys + off)
            Ps.append(pinned)
            Bs.append(torch.full((X.shape[0],), m, dtype=torch.int32, device="cuda"))
            off += X.shape[0]
        X, keys, d["pinned"], d["batch"] = torch.cat(Xs), torch.cat(Ks), torch.cat(Ps), torch.cat(Bs)
        d["mu"], d["lam"] = _lame(1e5, 0.45)
        d["u"] = 0.002 * torch.sin(3.0 * X.roll(1, 1))
        d["v"] = _uniform(g, X.shape, -0.05, 0.05)
    else:
        X, keys, d["pinned"], h = _mesh(g, case["nx"], case["ny"], case["nz"],
                                        "curve" if kind == "host" else case.get("order", "grid"))
        material = "per_tet" if kind == "rollout" else case.get("material", "uniform")
        d["mu"], d["lam"] = _material(g, material, case.get("model", "stvk"), keys.shape[0])
        d["u"] = _displacement(g, X, h, 0.05 if kind in ("map", "host", "assembled") else 0.01)
        d["w"] = _uniform(g, X.shape, -1.0, 1.0)
        d["v"] = 0.05 * d["w"]
        d["m"] = _uniform(g, (X.shape[0],), 0.5, 1.5) * RHO * h ** 3
        if kind == "springs":
            d["u"], d["v"] = 0.2 * h * d["w"], torch.zeros_like(X)
    d["X"], d["keys"] = X, keys
    return d


_DTYPE = {"f64": torch.float64, "f32": torch.float32, "f32x4": torch.float32}
_MODEL = {"stvk": abi.EBB_STVK, "nh": abi.EBB_NEOHOOKEAN}
_REDUCE = {"auto": abi.EBB_REDUCE_AUTO, "ordered": abi.EBB_REDUCE_TILED_ORDERED}


def _planes(x, dtype=torch.float64):
    """(N, 3) values as a field of 3 planes."""
    return x.T.to(dtype).contiguous()


def _bind(dm, name, x, precision):
    """Bind (N, 3) values as a vertex field of the precision's layout; the tensor."""
    if precision == "f32x4":
        t = torch.zeros((x.shape[0], 4), dtype=torch.float32, device="cuda")
        t[:, :3] = x
        abi.ebb_field_bind(dm.ctx, dm.verts, name, t, x4=True)
        return t
    return dm.bind(name, _planes(x, _DTYPE[precision]))


def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    per_tet = torch.is_tensor(d["mu"])
    dm = DeviceTetMesh(d["X"].cpu().numpy(), d["keys"].cpu().numpy(), d["mu"].cpu().numpy() if per_tet else None,
                       d["lam"].cpu().numpy() if per_tet else None, edges=kind in ("assembled", "springs"),
                       batch=d["batch"].cpu().numpy() if kind == "batch" else None)
    mu, lam = (0.0, 0.0) if per_tet else (d["mu"], d["lam"])
    s = {"kind": kind, "dm": dm, "case": dict(case)}
    precision = case.get("precision", "f64")
    model = _MODEL[case.get("model", "nh" if kind == "batch" else "stvk")]
    prec = abi.EBB_PREC_F64 if precision == "f64" else abi.EBB_PREC_F32
    if kind in ("map", "assembled"):
        s["u"] = _bind(dm, "u", d["u"], precision)
        s["w"] = _bind(dm, "w", d["w"], precision)
        s["f"] = _bind(dm, "f", torch.zeros_like(d["u"]), precision)
        s["Kw"] = _bind(dm, "Kw", torch.zeros_like(d["u"]), precision)
        s["opts"] = abi.map_opts(model, mu, lam, prec, _REDUCE[case.get("reduce", "auto")], abi.EBB_MAP_ZERO_OUT)
    elif kind in ("step", "batch"):
        s["u0"], s["v0"] = _planes(d["u"]), _planes(d["v"])
        s["u"], s["v"] = dm.bind("u", s["u0"].clone()), dm.bind("v", s["v0"].clone())
        dm.bind("pinned", d["pinned"])
        s["params"] = abi.step_params(model, DT, RHO, mu, lam, (0.0, 0.0, GZ), prec,
                                      max_iters=case.get("max_iters", 1000), rtol=case.get("rtol", 1e-8))
    elif kind == "rollout":
        dm.bind("pinned", d["pinned"])
        s["leaves"] = [_planes(d["u"]), _planes(d["v"]), d["mu"], d["lam"]]
        for t in s["leaves"]:
            t.requires_grad_(True)
        s["params"] = abi.step_params(model, DT, RHO, mu, lam, (0.0, 0.0, GZ), prec, max_iters=4000, rtol=1e-12)
    elif kind == "springs":
        dm.bind("X", _planes(d["X"], _DTYPE[precision]))
        abi.ebb_springs_init(dm.ctx, dm.tets, "X")
        s["q0"], s["v0"] = _planes(d["X"] + d["u"], _DTYPE[precision]), _planes(d["v"], _DTYPE[precision])
        s["q"], s["qd"] = dm.bind("q", s["q0"].clone()), dm.bind("qd", s["v0"].clone())
        dm.bind("m", d["m"].to(_DTYPE[precision]))
    else:
        s["fields"] = [_bind(dm, name, torch.zeros_like(d["u"]), "f32x4") for name in ("u", "w", "f", "Kw")]
        for name in ("u", "w", "f", "Kw"):
            s[name] = torch.zeros(d["u"].shape, dtype=torch.float32, pin_memory=True)
        s["u"].copy_(d["u"])
        s["w"].copy_(d["w"])
        s["opts"] = abi.map_opts(model, mu, lam, abi.EBB_PREC_F32, abi.EBB_REDUCE_AUTO,
                                 abi.EBB_MAP_ZERO_OUT | abi.EBB_MAP_HOST_XYZ)
    return s


# ---- one pass ------------------------------------------------------------------


def run(s):
    dm, kind, case = s["dm"], s["kind"], s["case"]
    if kind == "map":
        if case["ops"] == "fused":
            abi.ebb_map_tet_force_Kv(dm.ctx, dm.tets, "u", "w", "f", "Kw", s["opts"])
            return {"f": s["f"], "Kw": s["Kw"]}
        if case["ops"] == "kv":
            abi.ebb_map_tet_Kv(dm.ctx, dm.tets, "u", "w", "Kw", s["opts"])
            return {"Kw": s["Kw"]}
        abi.ebb_map_tet_forces(dm.ctx, dm.tets, "u", "f", s["opts"])
        return {"f": s["f"]}
    if kind in ("step", "batch"):
        s["u"].copy_(s["u0"])
        s["v"].copy_(s["v0"])
        if kind == "step":
            abi.ebb_cg_implicit_step(dm.ctx, dm.tets, "u", "v", "pinned", s["params"])
        else:
            abi.ebb_cg_implicit_step_batched(dm.ctx, dm.tets, "u", "v", "pinned", "batch", case["count"], s["params"])
        return {"u": s["u"], "v": s["v"]}
    if kind == "rollout":
        uT, vT = rollout(dm, *s["leaves"], case["steps"], s["params"], case["every"])
        grads = torch.autograd.grad((uT * uT).sum(), s["leaves"])
        return {"u": uT, "v": vT, "gu": grads[0], "gv": grads[1], "gmu": grads[2], "glam": grads[3]}
    if kind == "assembled":
        abi.ebb_assemble_tet_K(dm.ctx, dm.tets, "u", s["opts"])
        abi.ebb_spmv_tet_K(dm.ctx, dm.tets, "w", "Kw", s["opts"])
        return {"Kw": s["Kw"]}
    if kind == "springs":
        s["q"].copy_(s["q0"])
        s["qd"].copy_(s["v0"])
        energy = abi.ebb_springs_run(dm.ctx, dm.tets, "q", "qd", "m", SPRING_K, SPRING_DT, case["steps"], energy=True)
        return {"q": s["q"], "qd": s["qd"], "energy": energy}
    abi.ebb_map_tet_force_Kv_host(dm.ctx, dm.tets, "u", "w", "f", "Kw", s["u"], s["w"], s["f"], s["Kw"], s["opts"])
    return {"f": s["f"], "Kw": s["Kw"]}


# ---- what a pass cannot do without ---------------------------------------------


def work(case):
    kind = case["kind"]
    if kind == "batch":
        nt = sum(5 * n ** 3 for n in _sides(case))
        nv = sum((n + 1) ** 3 for n in _sides(case))
    else:
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        nt, nv = 5 * nx * ny * nz, (nx + 1) * (ny + 1) * (nz + 1)
    e = 8 if case.get("precision", "f64" if kind == "rollout" else "f32") == "f64" else 4
    per_tet = kind == "rollout" or case.get("material") == "per_tet"
    # keys, Dm^-1, V and the material; one K w product's (or force's) arithmetic in scalar operations
    tet, product, force = 16 + e * (12 if per_tet else 10), 300, 200
    if kind in ("map", "host"):
        ops = case.get("ops", "fused")
        fields = {"fused": 4, "kv": 3, "force": 2}[ops]
        flops = {"fused": product + 120, "kv": product, "force": force}[ops]
        # the host form reads and writes host memory; its fields still cross the device's
        return {"bytes": nt * tet + nv * 3 * e * fields, "flops": nt * flops}
    if kind == "assembled":
        return {"bytes": nt * tet + nv * (3 * e * 3 + ASSEMBLED_ROW * (9 * e + 4)),
                "flops": nt * 600 + nv * ASSEMBLED_ROW * 18}
    if kind == "springs":
        springs = nv * 12
        return {"bytes": case["steps"] * (springs * (4 + e) + nv * 13 * e), "flops": case["steps"] * springs * 20}
    # implicit steps: about this many CG iterations each; an iteration reads the tets once, p, and updates
    # the solver's FP64 vectors
    its = 12 if nt < 20000 else 30
    step = {"bytes": its * (nt * tet + nv * (3 * e * 2 + 3 * 8 * 8)) + nt * tet + nv * 4 * 24,
            "flops": its * (nt * product + nv * 48) + nt * 500}
    if kind == "rollout":   # forward, the replay between checkpoints, and one adjoint solve a step
        return {k: x * case["steps"] * 3 for k, x in step.items()}
    return step


# ---- the same in plain float64 -------------------------------------------------


class _Reference:
    """Linear tetrahedra in float64: forces, K w, the implicit step and its gradient."""

    def __init__(self, X, keys, model):
        self.k, self.model, self.nv = keys.long(), model, X.shape[0]
        x = X[self.k]
        Dm = (x[:, 1:] - x[:, :1]).transpose(1, 2)
        self.B, self.V = torch.linalg.inv(Dm), torch.linalg.det(Dm) / 6.0

    def grad(self, a):
        """The gradient (N_t, 3, 3) of a vertex field (N_v, 3)."""
        a = a[self.k]
        return (a[:, 1:] - a[:, :1]).transpose(1, 2) @ self.B

    def scatter(self, P, sign):
        """Sum of sign * V P b_a over the corners of every vertex."""
        H = (sign * self.V).reshape(-1, 1, 1) * (P @ self.B.transpose(1, 2))
        c = torch.cat([-H.sum(2, keepdim=True), H], 2).transpose(1, 2).reshape(-1, 3)
        return torch.zeros((self.nv, 3), dtype=torch.float64, device="cuda").index_add(0, self.k.reshape(-1), c)

    def state(self, u, mu, lam):
        G = self.grad(u)
        eye = torch.eye(3, dtype=torch.float64, device="cuda")
        F = G + eye
        mu, lam = (x.reshape(-1, 1, 1) if torch.is_tensor(x) else x for x in (mu, lam))
        if self.model == "stvk":
            E = 0.5 * (G + G.transpose(1, 2) + G.transpose(1, 2) @ G)
            tr = E.diagonal(dim1=1, dim2=2).sum(1).reshape(-1, 1, 1)
            return {"F": F, "S": 2 * mu * E + lam * tr * eye, "mu": mu, "lam": lam, "eye": eye}
        A = torch.linalg.inv(F).transpose(1, 2)
        lnJ = torch.log(torch.linalg.det(F)).reshape(-1, 1, 1)
        return {"F": F, "A": A, "lnJ": lnJ, "mu": mu, "lam": lam}

    def force(self, s):
        P = s["F"] @ s["S"] if self.model == "stvk" else s["mu"] * (s["F"] - s["A"]) + s["lam"] * s["lnJ"] * s["A"]
        return self.scatter(P, -1.0)

    def product(self, s, w):
        dF = self.grad(w)
        if self.model == "stvk":
            W = s["F"].transpose(1, 2) @ dF
            tr = W.diagonal(dim1=1, dim2=2).sum(1).reshape(-1, 1, 1)
            dP = dF @ s["S"] + s["F"] @ (s["mu"] * (W + W.transpose(1, 2)) + s["lam"] * tr * s["eye"])
        else:
            A = s["A"]
            tr = (A * dF).sum((1, 2)).reshape(-1, 1, 1)
            dP = s["mu"] * dF + (s["mu"] - s["lam"] * s["lnJ"]) * (A @ dF.transpose(1, 2) @ A) + s["lam"] * tr * A
        return self.scatter(dP, 1.0)

    def mass(self):
        q = (0.25 * RHO * self.V).repeat_interleave(4)
        return torch.zeros(self.nv, dtype=torch.float64, device="cuda").index_add(0, self.k.reshape(-1), q)[:, None]

    def solve(self, s, b, free, m):
        """A y = b on the free rows by conjugate gradients scaled by the mass and a stiffness per vertex."""
        lam = s["lam"] if torch.is_tensor(s["lam"]) else torch.full((self.k.shape[0], 1, 1), s["lam"],
                                                                     dtype=torch.float64, device="cuda")
        stiff = (lam.reshape(-1) * self.V * (self.B * self.B).sum((1, 2))).repeat_interleave(4)
        d = m + DT * DT * torch.zeros(self.nv, dtype=torch.float64, device="cuda").index_add(
            0, self.k.reshape(-1), stiff)[:, None]
        y, r = torch.zeros_like(b), b * free
        z = r / d
        p, rz, bb = z, (r * z).sum(), (r * r).sum()
        for it in range(2000):
            q = free * (m * p + DT * DT * self.product(s, p))
            a = rz / (p * q).sum()
            y, r = y + a * p, r - a * q
            if it % 5 == 4 and float((r * r).sum()) <= 1e-28 * float(bb):
                break
            z = r / d
            rz, old = (r * z).sum(), rz
            p = z + (rz / old) * p
        return y

    def rhs(self, s, v, m):
        g = torch.tensor([0.0, 0.0, GZ], dtype=torch.float64, device="cuda")
        return DT * (self.force(s) + m * g - DT * self.product(s, v))

    def step(self, u, v, mu, lam, free, m):
        s = self.state(u, mu, lam)
        v = v + self.solve(s, self.rhs(s, v, m), free, m)
        return u + DT * v, v


def _exact_rollout(case, d):
    ref = _Reference(d["X"], d["keys"], "stvk")
    free, m = (d["pinned"] == 0).double()[:, None], ref.mass()
    states = [(d["u"], d["v"])]
    for _ in range(case["steps"]):
        states.append(ref.step(*states[-1], d["mu"], d["lam"], free, m))
    uT, vT = states[-1]
    gu, gv, gmu, glam = 2 * uT, torch.zeros_like(vT), torch.zeros_like(d["mu"]), torch.zeros_like(d["lam"])
    for (u, v), (_, vn) in zip(reversed(states[:-1]), reversed(states[1:])):
        gn = gv + DT * gu
        lv = ref.solve(ref.state(u, d["mu"], d["lam"]), gn, free, m)
        leaves = [t.detach().clone().requires_grad_(True) for t in (u, v, d["mu"], d["lam"])]
        s = ref.state(leaves[0], leaves[2], leaves[3])
        dv = vn - v
        phi = (lv * (ref.rhs(s, leaves[1], m) - m * dv - DT * DT * ref.product(s, dv))).sum()
        a, b, c, e = torch.autograd.grad(phi, leaves)
        gu, gv, gmu, glam = gu + a, gn + b, gmu + c, glam + e
    return {"u": uT.T, "v": vT.T, "gu": gu.T, "gv": gv.T, "gmu": gmu, "glam": glam}


def _exact_springs(case, d):
    dt = _DTYPE[case["precision"]]
    X, q, qd, m = (t.to(dt).double() for t in (d["X"], d["X"] + d["u"], d["v"], d["m"]))
    k = d["keys"].long()
    pairs = torch.cat([k[:, [a, b]] for a in range(4) for b in range(4) if a != b])
    pairs = torch.unique(pairs[:, 0] * X.shape[0] + pairs[:, 1])
    i, j = pairs // X.shape[0], pairs % X.shape[0]
    L = (X[i] - X[j]).norm(dim=1, keepdim=True)
    for _ in range(case["steps"]):
        dq = q[i] - q[j]
        f = torch.zeros_like(q).index_add(0, i, SPRING_K * (L / dq.norm(dim=1, keepdim=True) - 1.0) * dq)
        a = f / m[:, None]
        q, qd = q + qd * SPRING_DT + 0.5 * a * SPRING_DT ** 2, qd + a * SPRING_DT
    return {"q": q.T, "qd": qd.T, "energy": float((0.5 * m[:, None] * qd * qd).sum())}


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "springs":
        return _exact_springs(case, d)
    if kind == "rollout":
        return _exact_rollout(case, d)
    ref = _Reference(d["X"], d["keys"], case.get("model", "nh"))
    if kind in ("step", "batch"):
        u, v = ref.step(d["u"], d["v"], d["mu"], d["lam"], (d["pinned"] == 0).double()[:, None], ref.mass())
        return {"u": u.T, "v": v.T}
    precision = case.get("precision", "f32x4" if kind == "host" else "f64")
    u, w = d["u"].to(_DTYPE[precision]).double(), d["w"].to(_DTYPE[precision]).double()
    s = ref.state(u, d["mu"], d["lam"])

    def laid_out(x):
        if kind == "host":
            return x
        return torch.nn.functional.pad(x, (0, 1)) if precision == "f32x4" else x.T

    out = {}
    if kind != "assembled" and case.get("ops", "fused") in ("fused", "force"):
        out["f"] = laid_out(ref.force(s))
    if kind == "assembled" or case.get("ops", "fused") in ("fused", "kv"):
        out["Kw"] = laid_out(ref.product(s, w))
    return out
