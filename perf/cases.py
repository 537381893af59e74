"""The measured work of the library: solves of hierarchical-P2 finite element systems on
box meshes, through the public entry points (`Handle`, `solve_batched`, the network's
training kernels).

Every system is assembled on the GPU with torch from the case's sizes and the seed: box
meshes of nx x ny x nz bricks cut into 6 Kuhn tetrahedra, interior vertices moved by a
seeded offset of at most `jitter` brick sizes, clamped at z = 0 (lid-driven for Stokes),
seeded loads.  The sizes, materials and tolerances are those of the repository's own
workloads (4^3 Laplacian, 32^3 elasticity, 24^3 Stokes, 40^3 mixed elasticity, batches of
boxes with n in 8..24) and of its tests (ragged boxes, FP64 and FP32 cycles, BF16 coarse
values, both saddle smoothers).
"""
import math

import numpy as np
import torch

from paper_1503_01287_gb300 import binding as B

DEV = torch.device("cuda" if torch.cuda.is_available() else "cpu")
SMOOTHERS = {"sgs": B.AMG_SMOOTHER_SGS, "bs": B.AMG_SMOOTHER_BS}
PRECISIONS = {"fp64": B.AMG_FP64, "fp32": B.AMG_FP32, "bf16": B.AMG_FP32_BF16}


def listed():
    return [
        # the smallest solve: a few thousand unknowns, where launches and latency are all
        {"name": "laplace_4_fp64", "do": "solve", "kind": "laplace", "nx": 4, "ny": 4, "nz": 4,
         "precision": "fp64", "jitter": 0.0, "tol": 1e-10},
        # a small part of odd sizes (a bracket, a unit cell), FP32 cycle
        {"name": "elasticity_7x5x11_fp32", "do": "solve", "kind": "elasticity", "nx": 7, "ny": 5,
         "nz": 11, "precision": "fp32", "jitter": 0.1, "tol": 1e-8},
        # an ordinary system with the library's default options (FP64 throughout)
        {"name": "elasticity_16_fp64", "do": "solve", "kind": "elasticity", "nx": 16, "ny": 16,
         "nz": 16, "precision": "fp64", "jitter": 0.0, "tol": 1e-8},
        # a ragged box with BF16 storage of the coarse operators
        {"name": "elasticity_25x19x22_bf16", "do": "solve", "kind": "elasticity", "nx": 25,
         "ny": 19, "nz": 22, "precision": "bf16", "jitter": 0.1, "tol": 1e-8},
        # the benchmark's elasticity system, with smoother weights set by the program
        {"name": "elasticity_32_fp32", "do": "solve", "kind": "elasticity", "nx": 32, "ny": 32,
         "nz": 32, "precision": "fp32", "jitter": 0.0, "tol": 1e-8, "ws": 0.9, "wc": 1.1},
        # a program whose matrix changes every step: setup and one solve
        {"name": "setup_solve_12x13x14_fp32", "do": "setup_solve", "kind": "elasticity",
         "nx": 12, "ny": 13, "nz": 14, "precision": "fp32", "jitter": 0.1, "tol": 1e-8},
        # the preconditioner inside a program's own Krylov method
        {"name": "precond_21x24x23_fp64", "do": "precond", "kind": "elasticity", "nx": 21,
         "ny": 24, "nz": 23, "precision": "fp64", "jitter": 0.1, "tol": 1e-8},
        # lid-driven Stokes flow, FP64 cycle
        {"name": "stokes_24_fp64", "do": "solve", "kind": "stokes", "nx": 24, "ny": 24, "nz": 24,
         "precision": "fp64", "jitter": 0.0, "tol": 1e-8, "smoother": "sgs", "restart": 300},
        # nearly incompressible elasticity, small and ragged, Braess-Sarazin smoother
        {"name": "mixed_13x11x15_bs_fp32", "do": "solve", "kind": "mixed", "nx": 13, "ny": 11,
         "nz": 15, "precision": "fp32", "jitter": 0.2, "tol": 1e-8, "nu": 0.49,
         "smoother": "bs", "restart": 100},
        # the largest: nearly incompressible elasticity, 1.66 M unknowns
        {"name": "mixed_40_fp32", "do": "solve", "kind": "mixed", "nx": 40, "ny": 40, "nz": 40,
         "precision": "fp32", "jitter": 0.2, "tol": 1e-8, "nu": 0.499, "smoother": "sgs",
         "restart": 300},
        # many parts, many loads: problems of different sizes side by side
        {"name": "batched_10x16_fp32", "do": "batched", "kind": "elasticity", "problems": 10,
         "nmin": 8, "nmax": 24, "rhs": 16, "precision": "fp32", "tol": 1e-8},
        # one step of training the weight network on its whole data set
        {"name": "weight_net_step_7560", "do": "train", "samples": 7560},
    ]


def _box(rng, lo, hi):
    """Brick counts of a box: a mean size spread over the logarithm, each axis near it."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return [max(lo, min(hi, round(n * rng.uniform(0.8, 1.25)))) for _ in range(3)]


def draw(rng):
    do = rng.choice(["solve", "solve", "solve", "saddle", "saddle", "setup_solve", "precond",
                     "batched", "train"])
    if do == "train":
        return {"do": do, "samples": round(math.exp(rng.uniform(math.log(200), math.log(7560))))}
    if do == "batched":
        lo = rng.randint(5, 12)
        return {"do": do, "kind": "elasticity", "problems": rng.randint(2, 8), "nmin": lo,
                "nmax": rng.randint(lo, 22), "rhs": rng.choice([1, 3, 5, 8, 16]),
                "precision": rng.choice(["fp32", "fp32", "fp64"]), "tol": 1e-8}
    if do == "saddle":
        nx, ny, nz = _box(rng, 5, 28)
        kind = rng.choice(["mixed", "stokes"])
        return {"do": "solve", "kind": kind, "nx": nx, "ny": ny, "nz": nz,
                "precision": "fp64" if kind == "stokes" else rng.choice(["fp32", "fp64"]),
                "jitter": 0.0 if kind == "stokes" else round(rng.uniform(0.02, 0.2), 3),
                "tol": 1e-8, "nu": round(0.5 - 10 ** rng.uniform(-3, -1.3), 5),
                "smoother": "sgs" if kind == "stokes" else rng.choice(["sgs", "bs"]),
                "restart": rng.choice([100, 200, 300])}
    nx, ny, nz = _box(rng, 4, 14 if do == "setup_solve" else 32)
    case = {"do": do, "kind": rng.choice(["laplace", "elasticity", "elasticity"]), "nx": nx,
            "ny": ny, "nz": nz, "precision": rng.choice(["fp64", "fp32", "fp32", "bf16"]),
            "jitter": round(rng.uniform(0.0, 0.15), 3), "tol": rng.choice([1e-8, 1e-10])}
    if do == "precond":
        case["precision"] = "fp64"
    if do == "solve" and rng.random() < 0.3:
        case["ws"] = round(rng.uniform(0.8, 1.1), 2)
        case["wc"] = round(rng.uniform(0.9, 1.3), 2)
    return case


# ------------------------------------------------------------------ mesh and assembly

PERMS = [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]
EDGES = [(0, 1), (1, 2), (2, 3), (0, 2), (0, 3), (1, 3)]   # local mid-side order


def _mesh(nx, ny, nz, lengths, jitter, rng):
    """Kuhn-split box: vertex coordinates, lattice indices, tetrahedra (brick-major),
    edges sorted by (min, max) vertex, and the 10 P2 nodes of every tetrahedron."""
    n = np.array([nx, ny, nz])
    k, j, i = np.meshgrid(np.arange(nz + 1), np.arange(ny + 1), np.arange(nx + 1), indexing="ij")
    grid = np.stack([i.ravel(), j.ravel(), k.ravel()], 1)
    h = np.array(lengths, dtype=np.float64) / n
    coords = grid * h
    if jitter > 0:
        off = rng.uniform(-jitter, jitter, coords.shape) * h
        off[(grid == 0) | (grid == n)] = 0.0
        coords = coords + off
    coords = torch.from_numpy(coords).to(DEV)
    grid = torch.from_numpy(grid).to(DEV)
    k, j, i = torch.meshgrid(torch.arange(nz, device=DEV), torch.arange(ny, device=DEV),
                             torch.arange(nx, device=DEV), indexing="ij")
    base = torch.stack([i.ravel(), j.ravel(), k.ravel()], 1)
    stride = torch.tensor([1, nx + 1, (nx + 1) * (ny + 1)], device=DEV)
    v0 = (base * stride).sum(1)
    tets = torch.stack([torch.stack([v0, v0 + stride[p[0]], v0 + stride[p[0]] + stride[p[1]],
                                     v0 + stride.sum()], 1) for p in PERMS], 1).reshape(-1, 4)
    nv = coords.shape[0]
    pairs = tets[:, torch.tensor(EDGES, device=DEV)]
    key = pairs.amin(2) * nv + pairs.amax(2)
    ukey, inv = torch.unique(key.reshape(-1), return_inverse=True)
    edges = torch.stack([ukey // nv, ukey % nv], 1)
    nodes = torch.cat([tets, inv.reshape(-1, 6) + nv], 1)
    return {"n": n, "coords": coords, "grid": grid, "tets": tets, "edges": edges,
            "nodes": nodes, "nv": nv, "nn": nv + edges.shape[0]}


def _gather_sum(vals, order, start, count):
    """Sum of each group's values in the order of the stable sort (the same bits always)."""
    out = torch.zeros((len(count),) + vals.shape[1:], dtype=vals.dtype, device=vals.device)
    for t in range(int(count.max())):
        m = torch.nonzero(count > t).squeeze(1)
        out[m] += vals[order[start[m] + t]]
    return out


def _csr(rows, cols, vals, nrows, ncols):
    """CSR of summed element entries; pattern kept where values are zero."""
    key = rows * ncols + cols
    key, order = torch.sort(key, stable=True)
    ukey, count = torch.unique_consecutive(key, return_counts=True)
    start = torch.cumsum(count, 0) - count
    rowptr = torch.zeros(nrows + 1, dtype=torch.int64, device=key.device)
    rowptr[1:] = torch.cumsum(torch.bincount(ukey // ncols, minlength=nrows), 0)
    out = _gather_sum(vals, order, start, count)
    return rowptr.int(), (ukey % ncols).int(), out


def _elements(mesh):
    """Gradient coefficients c[t, i, p] (grad phi_i = sum_p lambda_p c[t, i, p]) of the 10
    basis functions and the products int lambda_p lambda_q."""
    X = mesh["coords"][mesh["tets"]]
    J = X[:, 1:] - X[:, :1]
    inv = torch.linalg.inv(J)                       # grad lambda_k = column k - 1
    g = torch.empty(len(X), 4, 3, dtype=torch.float64, device=DEV)
    g[:, 1:] = inv.transpose(1, 2)
    g[:, 0] = -g[:, 1:].sum(1)
    vol = torch.linalg.det(J).abs() / 6
    c = torch.zeros(len(X), 10, 4, 3, dtype=torch.float64, device=DEV)
    for i in range(4):
        c[:, i] = g[:, i, None]
    for e, (a, b) in enumerate(EDGES):
        c[:, 4 + e, a] += 4 * g[:, b]
        c[:, 4 + e, b] += 4 * g[:, a]
    M = (torch.ones(4, 4, dtype=torch.float64, device=DEV)
         + torch.eye(4, dtype=torch.float64, device=DEV)) * (vol / 20)[:, None, None]
    return c, M


def _lame(nu, E=1.0):
    return E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))


def _velocity(mesh, kind, c, M, mu, lam):
    T = len(c)
    c30 = c.transpose(2, 3).reshape(T, 30, 4)
    G = (c30 @ M @ c30.transpose(1, 2)).reshape(T, 10, 3, 10, 3).permute(0, 1, 3, 2, 4)
    S = G.diagonal(dim1=3, dim2=4).sum(-1)[..., None, None] * torch.eye(
        3, dtype=torch.float64, device=DEV)
    if kind == "laplace":
        K = S
    elif kind == "elasticity":
        K = mu * S + mu * G.transpose(3, 4) + lam * G
    else:
        K = mu * S + mu * G.transpose(3, 4)
    K = 0.5 * (K + K.permute(0, 2, 1, 4, 3))
    tn = mesh["nodes"]
    rows = tn[:, :, None].expand(-1, 10, 10).reshape(-1)
    cols = tn[:, None, :].expand(-1, 10, 10).reshape(-1)
    return _csr(rows, cols, K.reshape(-1, 9), mesh["nn"], mesh["nn"])


def _rows_of(rowptr):
    n = len(rowptr) - 1
    return torch.repeat_interleave(torch.arange(n, device=rowptr.device),
                                   (rowptr[1:] - rowptr[:-1]).long())


def _matvec(rowptr, col, val, x):
    """y = A x for 3 x 3 blocks, x of shape (n, 3)."""
    n = len(rowptr) - 1
    A = torch.sparse_bsr_tensor(rowptr, col, val.reshape(-1, 3, 3), size=(3 * n, 3 * n))
    return (A @ x.reshape(-1, 1)).reshape(-1, 3)


def _traction(mesh, rng, count, gaussian):
    """`count` loads: a constant seeded traction on every triangle of z = 1."""
    top = mesh["grid"][:, 2] == mesh["n"][2].item()
    tets, nv = mesh["tets"], mesh["nv"]
    tris = []
    for d in range(4):
        t = tets[:, [q for q in range(4) if q != d]]
        tris.append(t[top[t].all(1)])
    tri = torch.unique(torch.sort(torch.cat(tris), 1).values, dim=0)
    X = mesh["coords"][tri]
    area = 0.5 * torch.linalg.norm(torch.linalg.cross(X[:, 1] - X[:, 0], X[:, 2] - X[:, 0]),
                                   dim=1)
    ekey = mesh["edges"][:, 0] * nv + mesh["edges"][:, 1]
    mids = torch.stack([torch.searchsorted(ekey, tri[:, a] * nv + tri[:, b])
                        for a, b in ((0, 1), (1, 2), (0, 2))], 1) + nv
    node = torch.cat([tri, mids], 1).reshape(-1)      # hats and bubbles integrate to |F|/3
    order = torch.sort(node, stable=True)
    ids, cnt = torch.unique_consecutive(order.values, return_counts=True)
    start = torch.cumsum(cnt, 0) - cnt
    out = torch.zeros(count, mesh["nn"], 3, dtype=torch.float64, device=DEV)
    for r in range(count):
        t = rng.standard_normal((len(tri), 3)) if gaussian else rng.uniform(-1, 1, (len(tri), 3))
        w = (area[:, None] / 3 * torch.from_numpy(t).to(DEV)).repeat_interleave(6, 0)
        out[r, ids] = _gather_sum(w, order.indices, start, cnt)
    return out


def _system(kind, nx, ny, nz, seed, jitter=0.0, lengths=(1.0, 1.0, 1.0), nu=0.3, n_rhs=1,
            gaussian=False):
    """The device arrays of one system and its right-hand sides (n_rhs, unknowns)."""
    rng = np.random.default_rng(seed)
    mesh = _mesh(nx, ny, nz, lengths, jitter, rng)
    c, M = _elements(mesh)
    lam, mu = (1.0, 1.0) if kind in ("laplace", "stokes") else _lame(nu)
    rowptr, col, val = _velocity(mesh, kind, c, M, mu, lam)
    grid, nv, nn = mesh["grid"], mesh["nv"], mesh["nn"]
    if kind == "stokes":
        fixed_v = ((grid == 0) | (grid == torch.from_numpy(mesh["n"]).to(DEV))).any(1)
        f = torch.zeros(n_rhs, nn, 3, dtype=torch.float64, device=DEV)
    else:
        fixed_v = grid[:, 2] == 0
        f = _traction(mesh, rng, n_rhs, gaussian)
    fixed = torch.cat([fixed_v, fixed_v[mesh["edges"]].all(1)])
    tags = torch.zeros(nn, dtype=torch.int32, device=DEV)
    tags[nv:] = 1
    tags[fixed] |= 0x10
    lift = torch.zeros(nn, 3, dtype=torch.float64, device=DEV)
    if kind == "stokes":        # the lid z = 1 moves in a seeded direction
        a = rng.uniform(0, 2 * math.pi)
        lid = torch.nonzero(grid[:, 2] == nz).squeeze(1)
        lift[lid, 0], lift[lid, 1] = math.cos(a), math.sin(a)
        ends = (grid[mesh["edges"], 2] == nz).sum(1) == 1    # u = 0 at a wall edge's middle
        lift[nv:][ends & fixed[nv:]] = -0.5 * lift[lid[0]]
        f = f - _matvec(rowptr, col, val, lift)
    f[:, fixed] = 0.0
    rows = _rows_of(rowptr)
    touch = fixed[rows] | fixed[col.long()]
    val[touch] = 0.0
    val[touch & (rows == col)] = torch.eye(3, dtype=torch.float64, device=DEV).reshape(-1)
    s = {"kind": kind, "a": (rowptr, col, val.reshape(-1)), "tags": tags, "fixed": fixed,
         "rhs": f.reshape(n_rhs, -1)}
    if kind in ("mixed", "stokes"):
        tets, tn = mesh["tets"], mesh["nodes"]
        Be = -torch.einsum("tkp,tjpb->tkjb", M, c)
        brow = tets[:, :, None].expand(-1, 4, 10).reshape(-1)
        bcol = tn[:, None, :].expand(-1, 4, 10).reshape(-1)
        bp, bc, bv = _csr(brow, bcol, Be.reshape(-1, 3), nv, nn)
        crow = tets[:, :, None].expand(-1, 4, 4).reshape(-1)
        ccol = tets[:, None, :].expand(-1, 4, 4).reshape(-1)
        cp, cc, mass = _csr(crow, ccol, M.reshape(-1), nv, nv)
        br = _rows_of(bp)
        order = torch.arange(len(br), device=DEV)
        cnt = (bp[1:] - bp[:-1]).long()
        g = -_gather_sum((bv * lift[bc.long()]).sum(1), order, bp[:-1].long(), cnt)
        bv[fixed[bc.long()]] = 0.0
        s["weights"] = _gather_sum(mass, torch.arange(len(cc), device=DEV), cp[:-1].long(),
                                   (cp[1:] - cp[:-1]).long())
        if kind == "stokes":    # rows between boundary data only are dropped
            g[_gather_sum(bv.abs().sum(1), order, bp[:-1].long(), cnt) == 0] = 0.0
        s["b"] = (bp, bc, bv.reshape(-1))
        s["c"] = (cp, cc, mass * (0.0 if kind == "stokes" else 1 / lam))
        s["rhs"] = torch.cat([s["rhs"], g[None].expand(n_rhs, -1)], 1)
    s["rhs"] = s["rhs"].contiguous()
    return s


# ------------------------------------------------------------------ a user's program


def _handle(case, s):
    o = {"precision": PRECISIONS[case["precision"]]}
    if "smoother" in case:
        o["smoother"] = SMOOTHERS[case["smoother"]]
        o["gmres_restart"] = case["restart"]
    h = B.Handle(*s["a"], s["tags"], s["kind"], B.default_options(**o), b=s.get("b"),
                 c=s.get("c"), device_ptrs=True)
    if s["kind"] == "stokes":
        h.set_pressure_weights(s["weights"].cpu().numpy())
    if "ws" in case:            # smoother and correction weights on the finest level
        w = np.ones((h.n_levels, 3))
        w[0] = (case["ws"], case["wc"], 1.0)
        h.set_level_weights(w)
    return h


def _case_system(case, seed):
    return _system(case["kind"], case["nx"], case["ny"], case["nz"], seed, case["jitter"],
                   nu=case.get("nu", 0.3))


def _batch_systems(case, seed):
    """Boxes of n in nmin..nmax with sides U[1, 4] and nu U[0.2, 0.45], N(0, 1) tractions;
    the sizes belong to the case, the rest to the seed."""
    sizes = np.random.default_rng(case["problems"] * 1000 + case["nmax"])
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(case["problems"]):
        n = int(sizes.integers(case["nmin"], case["nmax"] + 1))
        lengths = tuple(rng.uniform(1.0, 4.0, 3))
        out.append(_system("elasticity", n, n, n, int(rng.integers(1 << 30)), 0.0, lengths,
                           rng.uniform(0.2, 0.45), case["rhs"], True))
    return out


def _train_data(case, seed):
    """Network parameters (Glorot), inputs in the features' ranges and targets."""
    rng = np.random.default_rng(seed)
    n = case["samples"]
    theta = np.concatenate([rng.standard_normal(1024) * math.sqrt(2 / 80), np.zeros(64),
                            rng.standard_normal(4096) * math.sqrt(2 / 128), np.zeros(64),
                            rng.standard_normal(64) * math.sqrt(2 / 65), np.zeros(1)])
    x = rng.uniform(-1, 2, (n, 16))
    t = 0.05 * rng.standard_normal(n)
    return [torch.from_numpy(a.astype(np.float32)).to(DEV) for a in (theta, x, t)]


def prepare(case, seed):
    if case["do"] == "train":
        theta, x, t = _train_data(case, seed)
        z = torch.zeros_like(theta)
        return {"case": case, "theta": theta, "x": x, "t": t, "y": torch.empty_like(t),
                "grad": z.clone(), "m": z.clone(), "v": z.clone(),
                "loss": torch.zeros(1, device=DEV), "start": theta.clone(),
                "stream": torch.cuda.current_stream().cuda_stream}
    if case["do"] == "batched":
        ss = _batch_systems(case, seed)
        return {"case": case, "h": [_handle(case, s) for s in ss],
                "b": [s["rhs"] for s in ss], "x": [torch.zeros_like(s["rhs"]) for s in ss]}
    s = _case_system(case, seed)
    st = {"case": case, "n3": 3 * len(s["tags"])}
    if case["do"] == "setup_solve":
        st["sys"] = s
    else:
        st["h"] = _handle(case, s)
    st["b"] = s["rhs"][0].clone()
    st["x"] = torch.zeros_like(st["b"])
    return st


def run(state):
    case = state["case"]
    if case["do"] == "train":
        s = state
        s["theta"].copy_(s["start"])
        s["m"].zero_()
        s["v"].zero_()
        B.mlp_forward(s["theta"], s["x"], s["y"], s["stream"])
        B.mlp_gradient(s["theta"], s["x"], s["t"], s["grad"], s["loss"], s["stream"])
        B.mlp_adam(s["theta"], s["grad"], s["m"], s["v"], 1, 1e-3, s["stream"])
        return {"y": s["y"], "grad": s["grad"], "loss": s["loss"], "m": s["m"], "v": s["v"],
                "theta": s["theta"]}
    if case["do"] == "batched":
        B.solve_batched(state["h"], state["b"], state["x"], case["rhs"], case["tol"])
        return list(state["x"])
    if case["do"] == "precond":
        state["h"].apply_preconditioner(state["b"], state["x"])
        return state["x"]
    if case["do"] == "setup_solve":
        h = _handle(case, state["sys"])
        h.solve(state["b"], state["x"], case["tol"], True)
        h.free()
    else:
        state["h"].solve(state["b"], state["x"], case["tol"], True)
    n3 = state["n3"]
    return {"u": state["x"][:n3], "p": state["x"][n3:]} if "smoother" in case else state["x"]


# ------------------------------------------------------------------ what a pass cannot do without


def _counts(nx, ny, nz):
    """Vertices, edges and the stored blocks of A, B and C of a Kuhn-split box: two nodes
    are coupled when their vertices span a vertex, edge, triangle or tetrahedron."""
    v = (nx + 1) * (ny + 1) * (nz + 1)
    e = (nx * (ny + 1) * (nz + 1) + (nx + 1) * ny * (nz + 1) + (nx + 1) * (ny + 1) * nz
         + nx * ny * (nz + 1) + nx * (ny + 1) * nz + (nx + 1) * ny * nz + nx * ny * nz)
    t = 6 * nx * ny * nz
    f = 1 - v + e + t
    return v, v + e, v + 7 * e + 12 * f + 6 * t, v + 4 * e + 3 * f, v + 2 * e


def _work_system(case, nx, ny, nz, rhs=1):
    v, nodes, a, b, c = _counts(nx, ny, nz)
    saddle = case["kind"] in ("mixed", "stokes")
    entries = 9 * a + (6 * b + c if saddle else 0)
    unknowns = 3 * nodes + (v if saddle else 0)
    # one read of the operator and of b, one write of x; one operator application
    return {"bytes": 76 * a + (28 * b + 12 * c if saddle else 0) + 16 * unknowns * rhs,
            "flops": 2 * entries * rhs}


def work(case):
    if case["do"] == "train":
        n = case["samples"]
        return {"bytes": 4 * (5313 * 6 + 18 * n), "flops": 2 * 5184 * 4 * n}
    if case["do"] == "batched":
        sizes = np.random.default_rng(case["problems"] * 1000 + case["nmax"])
        ns = [int(sizes.integers(case["nmin"], case["nmax"] + 1))
              for _ in range(case["problems"])]
        ws = [_work_system(case, n, n, n, case["rhs"]) for n in ns]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    return _work_system(case, case["nx"], case["ny"], case["nz"])


# ------------------------------------------------------------------ the same in plain torch, 64 bits


def _block_operator(s):
    rowptr, col, val = s["a"]
    n = len(rowptr) - 1
    A = torch.sparse_bsr_tensor(rowptr, col, val.reshape(-1, 3, 3), size=(3 * n, 3 * n))
    diag = _rows_of(rowptr) == col
    Dinv = torch.linalg.inv(val.reshape(-1, 3, 3)[diag])
    return A, Dinv


def _pcg(A, Dinv, b, tol=1e-13, maxit=6000):
    """Block-Jacobi CG in 64 bits on the columns of b (n, k), each with its own scalars."""
    def M(r):
        return (Dinv @ r.reshape(len(Dinv), 3, -1)).reshape(r.shape)
    x = torch.zeros_like(b)
    r, bn = b.clone(), b.norm(dim=0)
    z = M(r)
    p, rz = z.clone(), (r * z).sum(0)
    for it in range(maxit):
        q = A @ p
        a = rz / (p * q).sum(0).clamp_min(1e-300)
        x += a * p
        r -= a * q
        if it % 25 == 24 and bool((r.norm(dim=0) <= tol * bn).all()):
            return x
        z = M(r)
        new = (r * z).sum(0)
        p = z + new / rz.clamp_min(1e-300) * p
        rz = new
    return None


def _minres(s, b, tol=1e-12, maxit=12000):
    """MINRES with the preconditioner diag(block Jacobi, scaled pressure mass) on the saddle
    system [A B^T; B -C]; None where it does not reach the tolerance."""
    A, Dinv = _block_operator(s)
    n3 = A.shape[0]
    bp, bc, bv = s["b"]
    np_ = len(bp) - 1
    cols = (3 * bc.long()[:, None] + torch.arange(3, device=DEV)).reshape(-1).int()
    Bm = torch.sparse_csr_tensor(3 * bp, cols, bv, size=(np_, n3))
    rows = _rows_of(bp).repeat_interleave(3)
    Bt = torch.sparse_coo_tensor(torch.stack([cols.long(), rows]), bv,
                                 size=(n3, np_)).coalesce().to_sparse_csr()
    Cm = torch.sparse_csr_tensor(*s["c"], size=(np_, np_))
    on = _rows_of(s["c"][0]) == s["c"][1]
    sd = 1 / (s["weights"] + s["c"][2][on])      # 1 / (mass + C) scale of the pressure

    def K(x):
        u, p = x[:n3, None], x[n3:, None]
        return torch.cat([A @ u + Bt @ p, Bm @ u - Cm @ p])[:, 0]

    def M(r):
        return torch.cat([(Dinv @ r[:n3].reshape(-1, 3, 1)).reshape(-1), sd * r[n3:]])

    # preconditioned Lanczos with Givens rotations (Paige and Saunders)
    x = torch.zeros_like(b)
    v_old, v = torch.zeros_like(b), b.clone()
    z = M(v)
    g_old, g = 1.0, math.sqrt(float(v @ z))
    eta, s_old, s0, c_old, c0 = g, 0.0, 0.0, 1.0, 1.0
    w_old, w = torch.zeros_like(b), torch.zeros_like(b)
    start = g
    for _ in range(maxit):
        z = z / g
        q = K(z)
        d = float(q @ z)
        v_new = q - (d / g) * v - (g / g_old) * v_old
        z_new = M(v_new)
        g_new = math.sqrt(max(float(v_new @ z_new), 0.0))
        a0 = c0 * d - c_old * s0 * g
        a1 = math.hypot(a0, g_new)
        a2 = s0 * d + c_old * c0 * g
        a3 = s_old * g
        c_old, s_old = c0, s0
        c0, s0 = a0 / a1, g_new / a1
        w_new = (z - a3 * w_old - a2 * w) / a1
        x += c0 * eta * w_new
        eta *= -s0
        v_old, v, z, g_old, g, w_old, w = v, v_new, z_new, g, g_new, w, w_new
        if abs(eta) <= tol * start or g_new == 0.0:
            r = b - K(x)
            return x if float(r.norm() / b.norm()) < 1e-10 else None
    return None


def _mlp_exact(case, seed):
    theta, x, t = (a.double() for a in _train_data(case, seed))
    theta.requires_grad_(True)
    w1, b1, w2, b2, w3, b3 = torch.split(theta, [1024, 64, 4096, 64, 64, 1])
    y = torch.relu(torch.relu(x @ w1.reshape(64, 16).T + b1) @ w2.reshape(64, 64).T + b2) @ w3 + b3
    loss = ((y - t) ** 2).mean()
    (grad,) = torch.autograd.grad(loss, theta)
    m, v = 0.1 * grad, 0.001 * grad * grad
    new = theta.detach() - 1e-3 * (m / 0.1) / ((v / 0.001).sqrt() + 1e-8)
    return {"y": y.detach(), "grad": grad, "loss": loss.detach().reshape(1), "m": m, "v": v,
            "theta": new}


def exact(case, seed):
    if case["do"] == "train":
        return _mlp_exact(case, seed)
    if case["do"] == "precond":
        return None             # the cycle itself has no closed form
    if case["do"] == "batched":
        return [_pcg(*_block_operator(s), s["rhs"].T.contiguous()).T.contiguous()
                for s in _batch_systems(case, seed)]
    s = _case_system(case, seed)
    if case["kind"] not in ("mixed", "stokes"):
        return _pcg(*_block_operator(s), s["rhs"].T.contiguous())[:, 0]
    x = None if s["rhs"].shape[1] > 500_000 else _minres(s, s["rhs"][0])
    if x is None:
        return None
    n3 = 3 * len(s["tags"])
    # the stopping rule leaves the Stokes pressure loosely determined (its constant, and
    # the corner values without an equation): the velocity is compared
    return {"u": x[:n3], "p": None if case["kind"] == "stokes" else x[n3:]}
