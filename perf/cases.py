"""The workloads whose speed this repository answers for, as a user's program runs them.

Every case is a thin extruded tetrahedral mesh (unit square x [-H, 0], H = eps (1 + 0.5 sin 2 pi x
sin 2 pi y), hexes split into six tetrahedra, interior nodes jittered) and one call, or one short
sequence of calls, of the public API on it. Meshes and loads are made from the seed on the GPU; a
state is what the calling program holds before the call: the mesh on the host, the hierarchy on
the device, the right-hand sides on the device (or, for `host`, in page-locked host memory).

Kinds of case:
  solve    one right-hand side with the hierarchy resident (vemg_solve): the time step of an
           ocean model, which keeps the mesh and solves again and again
  host     the same with the vectors in host memory (vemg_solve_host)
  batch    k right-hand sides at once (vemg_solve_batch)
  engine   requests served by an engine of 8 slots: admitted, iterated two steps at a time, retired
  first    a new mesh: assembly, setup and the first solve (vemg_assemble, vemg_setup, vemg_solve),
           what a server pays on a request for a mesh that it has not seen
  load     a load vector b = M f from nodal values (vemg_load)
  spmv     one product with the operator (vemg_spmv), e.g. to check a residual
  precond  one application of the preconditioner (vemg_precond) inside the caller's own iteration
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_0912_1976_gb300 import vemg as V

PREC = {"fp64": V.VEMG_PREC_FP64, "fp32": V.VEMG_PREC_FP32, "bf16": V.VEMG_PREC_BF16}
BC = {"neumann": V.VEMG_NEUMANN, "dirichlet_top": V.VEMG_DIRICHLET_TOP}
PRECOND = {"additive": V.VEMG_PRECOND_ADDITIVE, "vl_sor": V.VEMG_PRECOND_VL_SOR, "sa": V.VEMG_PRECOND_SA}
MAX_IT = 1000


def _case(kind, nx, ny, nz, *, name=None, eps=1e-3, xy=0.0, bc="neumann", prec="fp64", precond="additive", k=1,
          rtol=1e-8):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "eps": eps, "xy": xy, "bc": bc, "prec": prec,
         "precond": precond, "k": k, "rtol": rtol}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest problem of this repository (its 16 x 16 x 8 thin box, 2,601 nodes) with the
        # default options: a solve is launches and latency
        _case("solve", 16, 16, 8, name="solve_box16_fp64", eps=1e-2, rtol=1e-10),
        # the 256 x 256 x 32 mesh of bench.py in the precision it runs by default: 2.2M nodes
        _case("solve", 256, 256, 32, name="solve_256_bf16", prec="bf16"),
        # a rigid-lid problem of medium size with odd extents, everything in FP64
        _case("solve", 131, 113, 25, name="solve_dirichlet_fp64", eps=1e-2, bc="dirichlet_top"),
        # a mesh that is unstructured in the horizontal too, with the {1, x, y} surface chain that
        # such meshes take, FP32 cycles
        _case("solve", 96, 90, 24, name="solve_unstructured_fp32", eps=1e-2, xy=0.2, prec="fp32"),
        # the caller's vectors in host memory, SA on A (the comparison preconditioner)
        _case("host", 70, 61, 18, name="host_sa_fp32", eps=1e-2, prec="fp32", precond="sa"),
        # 64 right-hand sides on 3.7M nodes: the largest batch
        _case("batch", 384, 384, 24, name="batch64_384_fp32", prec="fp32", k=64),
        # an odd number of right-hand sides on a mesh of the serving stream
        _case("batch", 134, 134, 24, name="batch5_134_bf16", prec="bf16", k=5),
        # a served mix on one mesh: 8 requests in 8 slots
        _case("engine", 100, 100, 24, name="engine8_100_fp64", eps=1e-2, k=8, prec="fp64"),
        # the bench mesh, cold: assembly, setup, first solve
        _case("first", 256, 256, 32, name="first_256_bf16", prec="bf16"),
        # the smallest mesh of the serving stream, cold, rigid lid
        _case("first", 44, 44, 24, name="first_44_fp32", eps=1e-1, bc="dirichlet_top", prec="fp32"),
        # a product with the operator, 1M nodes, odd extents
        _case("spmv", 211, 197, 24, name="spmv_211"),
        # the FP64 preconditioner, 0.5M nodes
        _case("precond", 150, 141, 24, name="precond_150_fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: meshes of 2,600 to 2.2M nodes (3.7M for a batch), the
    aspect ratios, boundary conditions, precisions and batch widths that the calls take in use."""
    kind = rng.choice(["solve", "solve", "solve", "host", "batch", "batch", "engine", "first", "load", "spmv",
                       "precond"])
    eps = rng.choice([1e-1, 1e-2, 1e-3])
    bc = rng.choice(["neumann", "neumann", "dirichlet_top"])
    prec = rng.choice(["fp64", "fp32", "bf16"])
    precond = rng.choice(["additive", "additive", "additive", "vl_sor", "sa"]) if kind in ("solve", "host") else "additive"
    xy = 0.0
    k = 1
    # nodes: 2,600 .. most, in a mesh of 8 .. 40 layers and 1:2 .. 2:1 extents
    most = {"engine": 4e5, "batch": 1.5e6}.get(kind, 2.1e6)
    n = math.exp(rng.uniform(math.log(2600.0), math.log(most)))
    nz = _log_int(rng, 8, 40)
    ratio = math.exp(rng.uniform(-0.5, 0.5))
    side = math.sqrt(n / (nz + 1))
    nx, ny = max(8, int(side * ratio)), max(8, int(side / ratio))
    if kind == "batch":
        k = min(64, max(2, min(_log_int(rng, 2, 64), int(1.6e7 / n))))
    if kind == "engine":
        k = rng.randint(1, 8)
    if kind in ("batch", "engine"):
        precond = "additive"
    if precond == "vl_sor":
        bc = "neumann"
    if precond == "sa":
        eps = rng.choice([1e-1, 1e-2])   # it slows down as the domain gets thinner (section 6)
    if kind in ("spmv", "load"):
        prec, bc = "fp64", "neumann"
    if kind == "precond":
        prec = "fp64"
    if kind == "solve" and bc == "neumann" and precond == "additive" and rng.random() < 0.25:
        xy, eps = 0.2, rng.choice([1e-1, 1e-2])
    return _case(kind, nx, ny, nz, eps=eps, xy=xy, bc=bc, prec=prec, precond=precond, k=k,
                 rtol=rng.choice([1e-8, 1e-9]))


# ---------------------------------------------------------------------------
# inputs

def _unit_tets():
    """The six tetrahedra of a hex as corner offsets (i, j, k), positively oriented for k downwards."""
    out = []
    for perm in itertools.permutations(range(3)):
        v = [np.zeros(3, dtype=np.int64)]
        for ax in perm:
            w = v[-1].copy()
            w[ax] += 1
            v.append(w)
        p = [np.array([a[0], a[1], -a[2]], dtype=np.float64) for a in v]
        if np.dot(p[1] - p[0], np.cross(p[2] - p[0], p[3] - p[0])) < 0:
            v[2], v[3] = v[3], v[2]
        out.append(v)
    return out


def _mesh(case, seed):
    """(xyz, tets, tags, top_tris) as GPU tensors. Node id = column * (nz + 1) + layer, top first."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(1_000_003 * int(seed) + 17)
    ncol, n = (nx + 1) * (ny + 1), (nx + 1) * (ny + 1) * (nz + 1)
    nid = torch.arange(n, device=dev)
    k, col = nid % (nz + 1), nid // (nz + 1)
    i, j = col % (nx + 1), col // (nx + 1)
    u = torch.rand((3, n), generator=g, device=dev, dtype=torch.float64) * 2.0 - 1.0
    coast = (i == 0) | (i == nx) | (j == 0) | (j == ny)
    inner = ((k > 0) & (k < nz)).double() * 0.3
    moved = (~coast).double() * case["xy"]

    hi = torch.arange(nx, device=dev)
    hj = torch.arange(ny, device=dev)
    hk = torch.arange(nz, device=dev)
    hj, hi, hk = (t.reshape(-1) for t in torch.meshgrid(hj, hi, hk, indexing="ij"))
    tets = torch.stack([torch.stack([((hj + int(c[1])) * (nx + 1) + hi + int(c[0])) * (nz + 1) + hk + int(c[2])
                                     for c in v], 1) for v in _unit_tets()], 1).reshape(-1, 4)
    while True:
        x = i.double() / nx + moved * u[0] / nx
        y = j.double() / ny + moved * u[1] / ny
        h = case["eps"] * (1.0 + 0.5 * torch.sin(2 * math.pi * x) * torch.sin(2 * math.pi * y))
        z = torch.where(k == 0, 0.0, -h * (k.double() - inner * u[2]) / nz)
        xyz = torch.stack([x, y, z], 1)
        p = xyz[tets]
        d = p[:, 1:] - p[:, :1]
        bad = (d[:, 0] * torch.linalg.cross(d[:, 1], d[:, 2])).sum(1) <= 0.0
        if not bool(bad.any()):
            break
        u[:, torch.unique(tets[bad])] *= 0.5   # a folded tetrahedron: its nodes move half as far
    qj, qi = (t.reshape(-1) for t in torch.meshgrid(torch.arange(ny, device=dev), torch.arange(nx, device=dev),
                                                    indexing="ij"))

    def top(a, b):
        return (b * (nx + 1) + a) * (nz + 1)

    v00, v10, v11, v01 = top(qi, qj), top(qi + 1, qj), top(qi + 1, qj + 1), top(qi, qj + 1)
    tris = torch.stack([torch.stack([v00, v10, v11], 1), torch.stack([v00, v11, v01], 1)], 1).reshape(-1, 3)
    tags = (k == 0).to(torch.uint8) + 2 * (k == nz).to(torch.uint8) + 4 * coast.to(torch.uint8)
    assert ncol * (nz + 1) == n
    return xyz, tets, tags, tris


def _loads(case, n, seed):
    """Independent N(0, 1) nodal loads, one row per right-hand side."""
    g = torch.Generator(device="cuda")
    g.manual_seed(7919 * int(seed) + 5)
    return torch.randn((case["k"], n), generator=g, device="cuda", dtype=torch.float64)


def _options(case):
    return V.vemg_default_options(bc=BC[case["bc"]], precision=PREC[case["prec"]], precond=PRECOND[case["precond"]],
                                  surf_nullspace=3 if case["xy"] > 0.0 else 1)


def prepare(case, seed):
    mesh = V.Mesh(*(t.cpu().numpy() for t in _mesh(case, seed)))
    st = {"case": case, "mesh": mesh, "b": _loads(case, mesh.n, seed)}
    kind = case["kind"]
    if kind not in ("first", "load"):
        A = V.vemg_assemble(mesh)
        st["h"] = V.vemg_setup(A, mesh, _options(case))
        if kind in ("batch", "engine", "host"):
            A.free()   # such a program keeps the hierarchy only
    if kind == "host":
        n = mesh.n
        b, x = (torch.empty(n, dtype=torch.float64, pin_memory=True) for _ in range(2))
        b.copy_(st.pop("b")[0])
        st["pinned"] = (b, x)
        st["bh"], st["xh"] = b.numpy(), x.numpy()
    if kind == "engine":
        st["engine"] = V.Engine(st["h"], 8)
        st["x"] = torch.empty_like(st["b"])
    if kind == "precond" and case["bc"] == "dirichlet_top":
        # its vectors hold the unknowns: the nodes below the top
        st["b"] = st["b"][:, : V.vemg_get_size(st["h"], "n") - V.vemg_get_size(st["h"], "mtop")].contiguous()
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------------------
# the calls

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        return V.vemg_solve(state["h"], state["b"][0], rtol=case["rtol"], max_it=MAX_IT)[0]
    if kind == "host":
        return V.vemg_solve_host(state["h"], state["bh"], state["xh"], rtol=case["rtol"], max_it=MAX_IT)[0]
    if kind == "batch":
        return V.vemg_solve_batch(state["h"], state["b"], rtol=case["rtol"], max_it=MAX_IT)[0]
    if kind == "engine":
        eng, x = state["engine"], state["x"]
        open_ = {eng.admit(b, rtol=case["rtol"], max_it=MAX_IT): c for c, b in enumerate(state["b"])}
        while open_:
            eng.launch(2)
            eng.wait()
            for slot in [s for s in open_ if eng.poll(s)[0] == V.VEMG_SLOT_DONE]:
                eng.retire(slot, x[open_.pop(slot)])
        return x
    if kind == "first":
        A = V.vemg_assemble(state["mesh"])
        h = V.vemg_setup(A, state["mesh"], _options(case))
        x = V.vemg_solve(h, state["b"][0], rtol=case["rtol"], max_it=MAX_IT)[0]
        state["kept"] = (A, h)   # in use from here on; the ones of the pass before are released
        # copies: A.tensors() are views of memory that goes with A
        rowptr, col, val = (t.clone() for t in A.tensors())
        return {"rowptr": rowptr, "col": col, "val": val, "x": x}
    if kind == "load":
        return V.vemg_load(state["mesh"], state["b"][0])
    if kind == "spmv":
        return V.vemg_spmv(state["h"], state["b"][0])
    return V.vemg_precond(state["h"], state["b"][0])


def work(case):
    """The operator, the loads and the result once; for a product or a load that is all there is to
    do, a solve comes back to the operator in each of its iterations. A cold start reads the mesh,
    and writes the operator too. Operations: a multiply-add per stored entry and right-hand side."""
    nx, ny, nz, k = case["nx"], case["ny"], case["nz"], case["k"]
    n = (nx + 1) * (ny + 1) * (nz + 1)
    # a Kuhn-split box: vertices + 2 (axis edges + face diagonals + body diagonals)
    edges = (nx * (ny + 1) * (nz + 1) + (nx + 1) * ny * (nz + 1) + (nx + 1) * (ny + 1) * nz
             + nx * ny * (nz + 1) + nx * (ny + 1) * nz + (nx + 1) * ny * nz + nx * ny * nz)
    nnz = n + 2 * edges
    mesh = 24.0 * n + 16.0 * 6 * nx * ny * nz
    matrix = 12.0 * nnz + 4.0 * (n + 1)
    if case["kind"] == "load":
        return {"bytes": mesh + 16.0 * n, "flops": 60.0 * 6 * nx * ny * nz}
    if case["kind"] == "first":
        return {"bytes": mesh + matrix + 16.0 * n, "flops": 200.0 * 6 * nx * ny * nz + 2.0 * nnz}
    return {"bytes": matrix + 16.0 * n * k, "flops": 2.0 * nnz * k}


# ---------------------------------------------------------------------------
# the same results in plain torch, 64 bits

def _stiffness(xyz, tets):
    """K_e[a][b] = integral grad N_a . grad N_b of every tetrahedron, and six times its volume."""
    p = xyz[tets]
    d = p[:, 1:] - p[:, :1]
    c1 = torch.linalg.cross(d[:, 1], d[:, 2])
    c2 = torch.linalg.cross(d[:, 2], d[:, 0])
    c3 = torch.linalg.cross(d[:, 0], d[:, 1])
    det = (d[:, 0] * c1).sum(1)
    c = torch.stack([-(c1 + c2 + c3), c1, c2, c3], 1)
    return c @ c.transpose(1, 2) / (6.0 * det)[:, None, None], det


def _operator(xyz, tets):
    n = xyz.shape[0]
    K, _ = _stiffness(xyz, tets)
    key = (tets[:, :, None] * n + tets[:, None, :]).reshape(-1)
    key, at = torch.unique(key, return_inverse=True)
    val = torch.zeros(key.numel(), dtype=torch.float64, device=xyz.device).index_add_(0, at, K.reshape(-1))
    row, col = key // n, key % n
    rowptr = torch.searchsorted(row, torch.arange(n + 1, device=xyz.device))
    return rowptr, row, col, val


def _solve(case, rowptr, row, col, val, b, limit=6000):
    """x of A x = b by conjugate gradients with the exact inverse of each column of nodes as the
    preconditioner, far below the tolerance of the case. b: (n, k)."""
    n, layers = b.shape[0], case["nz"] + 1
    dirichlet = case["bc"] == "dirichlet_top"
    if dirichlet:   # the top nodes leave the system: identity rows, zero right-hand side
        fixed = torch.arange(n, device=b.device) % layers == 0
        off = (fixed[row] | fixed[col])
        val = torch.where(off, torch.where(row == col, 1.0, 0.0), val)
        b = torch.where(fixed[:, None], 0.0, b)
    else:
        b = b - b.mean(0)
    A = torch.sparse_csr_tensor(rowptr, col, val, (n, n))
    blocks = torch.zeros((n // layers, layers, layers), dtype=torch.float64, device=b.device)
    own = row // layers == col // layers
    blocks[row[own] // layers, row[own] % layers, col[own] % layers] = val[own]
    inv = torch.linalg.inv(blocks)

    def precond(r):
        z = (inv @ r.reshape(n // layers, layers, -1)).reshape(n, -1)
        return z if dirichlet else z - z.mean(0)

    x, r = torch.zeros_like(b), b.clone()
    z = precond(r)
    p, rz = z, (r * z).sum(0)
    first = rz.clone()
    for it in range(limit):
        q = A @ p
        alpha = rz / (p * q).sum(0)
        x += alpha * p
        r -= alpha * q
        z = precond(r)
        new = (r * z).sum(0)
        if it % 20 == 0 and bool((new <= 1e-28 * first).all()):
            return x if dirichlet else x - x.mean(0)
        p = z + (new / rz) * p
        rz = new
    return None


def exact(case, seed):
    kind = case["kind"]
    n = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
    if kind == "precond" or n * case["k"] > 2_500_000:
        return None   # a method's own intermediate result; a batch that takes minutes this way
    xyz, tets, tags, _ = _mesh(case, seed)
    b = _loads(case, n, seed)
    if kind == "load":
        _, det = _stiffness(xyz[:, :], tets)
        f = b[0]
        fe = f[tets]
        out = torch.zeros_like(f)
        return out.index_add_(0, tets.reshape(-1), ((det / 120.0)[:, None] * (fe + fe.sum(1, keepdim=True))).reshape(-1))
    rowptr, row, col, val = _operator(xyz, tets)
    if kind == "spmv":
        # the single steps number the nodes top first, each group in the caller's order
        order = torch.cat([torch.nonzero(tags & 1).reshape(-1), torch.nonzero((tags & 1) == 0).reshape(-1)])
        x = torch.empty_like(b[0])
        x[order] = b[0]
        y = torch.zeros_like(x).index_add_(0, row, val * x[col])
        return y[order]
    x = _solve(case, rowptr, row, col, val, b.t().contiguous())
    x = None if x is None else x.t().contiguous()
    if kind == "first":
        return {"rowptr": rowptr.to(torch.int32), "col": col.to(torch.int32), "val": val, "x": None if x is None else x[0]}
    if kind in ("batch", "engine"):
        return x
    return None if x is None else (x[0].cpu().numpy() if kind == "host" else x[0])
