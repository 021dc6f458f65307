"""What the library is used for, as cases that can be timed and compared.

A user of this library assembles -div(sigma grad u) = f on a mesh, builds an
SA-AMG hierarchy of the matrix (`Hierarchy`), and solves: one right-hand side
(`solve`), several of one operator (`solve_batch`), one each of several
operators (`solve_group`, the serving loop's continuous batch); some apply the
V-cycle inside an iteration of their own (`vcycle`) or only want the strength
filter (`strength`).  The operators are the repository's workloads -- layered
squares and cubes (the serving operators), the battery stack, Voronoi regions
with rotated anisotropy, spherical inclusions, the two-domain study -- from
1e3 to 7e6 unknowns, in both solve forms and with both main measures.

The matrices are assembled on the device with torch: Q1 / trilinear elements
on a box, Dirichlet nodes eliminated symmetrically, 9 / 27-point rows.
"""
import math

import numpy as np
import torch

import paper_2602_05686_gb300 as sa

TOL = 1e-8                                       # the paper's residual reduction
THETA = {"material": 0.05, "classical": 0.04}    # the thresholds the workloads use
# V-cycles of a solve to TOL, roughly (from the workloads' measured counts): for work() only
CYCLES = {"layered": 15, "two_domain": 20, "battery": 15, "voronoi": 100, "inclusions": 38}


def listed():
    return [
        # the smallest call: one solve of the 32 x 32 layered square with a kept hierarchy (time stepping, a
        # parameter study); three levels of at most 1089 unknowns, so launches and their latency are the time
        dict(name="solve_layered2d_32", op="solve", kind="layered", dim=2, n=32, contrast=1e-4, measure="material",
             precision="fp64", max_coarse=64),
        # a new operator arrives at the server: setup and one solve.  2D, small enough to be solved directly
        dict(name="new_layered2d_64", op="setup_solve", kind="layered", dim=2, n=64, contrast=1e4,
             measure="material", precision="fp32", max_coarse=5000),
        # the same for a 3D operator of the middle of the serving range (118k unknowns)
        dict(name="new_layered3d_48", op="setup_solve", kind="layered", dim=3, n=48, contrast=1e4,
             measure="material", precision="fp32", max_coarse=5000),
        # the server's continuous batch: sixteen cached operators of different sizes, one request each
        dict(name="group16_fp32", op="group", kind="layered", m=16, n=14, contrast=1e3, measure="material",
             precision="fp32", max_coarse=5000),
        # the theta studies: a two-domain square, FP64, hierarchy kept
        dict(name="solve_two_domain_257", op="solve", kind="two_domain", dim=2, n=257, contrast=1e4,
             measure="material", precision="fp64", max_coarse=64),
        # one right-hand side of a 3D anisotropic operator in FP64 (material measure, about 1e6 unknowns)
        dict(name="solve_voronoi_101_fp64", op="solve", kind="voronoi", dim=3, n=101, measure="material",
             precision="fp64", max_coarse=5000),
        # the same operator family with the FP32 V-cycle and the classical measure
        dict(name="solve_voronoi_120_fp32", op="solve", kind="voronoi", dim=3, n=120, measure="classical",
             precision="fp32", max_coarse=5000),
        # the battery stack's preconditioner: build it and apply it once, as a user with a Krylov method of their
        # own does in every time step (contrast 1e10, stretched cells: many levels, long coarse rows)
        dict(name="precond_battery_80", op="setup_apply", kind="battery", dim=3, n=80, measure="material",
             precision="fp64", max_coarse=5000),
        # several load cases of one operator as a block, FP64: eight columns
        dict(name="batch8_inclusions_128_fp64", op="batch", kind="inclusions", dim=3, n=128, k=8,
             measure="classical", precision="fp64", max_coarse=5000),
        # the same in the FP32-V-cycle form on a larger grid
        dict(name="batch8_inclusions_160_fp32", op="batch", kind="inclusions", dim=3, n=160, k=8,
             measure="classical", precision="fp32", max_coarse=5000),
        # a whole large run: setup and one solve of 7.2e6 unknowns (the headline workload's operator)
        dict(name="new_inclusions_192", op="setup_solve", kind="inclusions", dim=3, n=192, measure="classical",
             precision="fp32", max_coarse=5000),
        # the material-aware strength filter alone, as a step of a caller's own coarsening (2.1e6 nodes)
        dict(name="strength_voronoi_128", op="strength", kind="voronoi", dim=3, n=128, measure="material"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    prec = rng.choice(("fp64", "fp32"))
    what = rng.choice(("solve2d", "solve3d", "new2d", "new3d", "group", "precond", "batch", "strength"))
    if what == "solve2d":
        kind = rng.choice(("layered", "two_domain"))
        return dict(op="solve", kind=kind, dim=2, n=_logint(rng, 24, 400), contrast=10.0 ** rng.uniform(2, 5),
                    measure="material", precision=prec, max_coarse=rng.choice((64, 500, 5000)))
    if what == "solve3d":
        return dict(op="solve", kind="voronoi", dim=3, n=_logint(rng, 24, 110),
                    measure=rng.choice(("material", "classical")), precision=prec, max_coarse=5000)
    if what == "new2d":
        return dict(op="setup_solve", kind="layered", dim=2, n=_logint(rng, 16, 512), contrast=10.0 ** rng.uniform(2, 5),
                    measure="material", precision=prec, max_coarse=5000)
    if what == "new3d":
        kind = rng.choice(("layered", "inclusions"))
        return dict(op="setup_solve", kind=kind, dim=3, n=_logint(rng, 20, 150), contrast=10.0 ** rng.uniform(2, 5),
                    measure="classical" if kind == "inclusions" else "material", precision=prec, max_coarse=5000)
    if what == "group":
        return dict(op="group", kind="layered", m=rng.randint(2, 20), n=rng.randint(10, 20),
                    contrast=10.0 ** rng.uniform(2, 4), measure="material", precision=prec, max_coarse=5000)
    if what == "precond":
        return dict(op="setup_apply", kind="battery", dim=3, n=_logint(rng, 20, 80), measure="material",
                    precision="fp64", max_coarse=5000)
    if what == "batch":
        return dict(op="batch", kind="inclusions", dim=3, n=_logint(rng, 32, 120), k=rng.randint(2, 8),
                    measure="classical", precision=prec, max_coarse=5000)
    return dict(op="strength", kind=rng.choice(("voronoi", "battery")), dim=3, n=_logint(rng, 20, 128),
                measure=rng.choice(("material", "classical")))


# ---------------------------------------------------------------------------
# operators
# ---------------------------------------------------------------------------
def _grid(case, gi=0):
    """Elements per axis (x, y, z; z = 0 in 2D) and cell sizes."""
    kind, n = case["kind"], case["n"]
    if case["op"] == "group":   # operator gi of a group: alternating 2D and 3D, sizes spread over the small serving range
        n = n + 2 * gi
        return ((n * 3, n * 3, 0), (1.0 / (n * 3),) * 2 + (1.0,)) if gi % 2 == 0 else ((n, n, n), (1.0 / n,) * 3)
    if case["dim"] == 2:
        return (n, n, 0), ((2.0 if kind == "two_domain" else 1.0) / n,) * 2 + (1.0,)
    if kind == "battery":
        return (n, n, 2 * n), (1.0 / n, 1.0 / n, 0.01 / n)
    return (n, n, n), (1.0 / n,) * 3


def _rotations(u):
    """Rotation matrices from rows of three uniforms (Shoemake's quaternions)."""
    a, b = np.sqrt(1 - u[:, 0]), np.sqrt(u[:, 0])
    x, y = a * np.sin(2 * np.pi * u[:, 1]), a * np.cos(2 * np.pi * u[:, 1])
    z, w = b * np.sin(2 * np.pi * u[:, 2]), b * np.cos(2 * np.pi * u[:, 2])
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                     2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                     2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)


def _tensors(case, el, rng, gi=0):
    """Packed conductivity per element, [components, elements] (elements x fastest)."""
    nx, ny, nz = el
    dim = 3 if nz else 2
    nzz = max(nz, 1)
    kind = case["kind"]
    dev = dict(device="cuda", dtype=torch.float64)
    diag = (0, 1, 2) if dim == 3 else (0, 1)
    K = torch.zeros((6 if dim == 3 else 3, nzz, ny, nx), **dev)
    if kind in ("layered", "battery"):
        # layers of conductivity along the last axis, each layer's value scattered a little
        m = nz if dim == 3 else ny
        cycle = (1.0, case["contrast"]) if kind == "layered" else (1e5, 1e-5, 1e2)
        w = 4 if kind == "layered" else 8
        lay = (np.arange(m) // w)
        s = np.asarray(cycle)[lay % len(cycle)] * rng.uniform(0.5, 2.0, lay[-1] + 1)[lay]
        s = torch.as_tensor(s, **dev)
        for c in diag:
            K[c] = s[:, None, None] if dim == 3 else s[None, :, None]
    elif kind == "two_domain":
        K[0] = 1.0
        K[0, :, :, nx // 2:] = case["contrast"] * rng.uniform(0.5, 2.0)
        K[1] = rng.uniform(0.5, 2.0)
    elif kind == "voronoi":
        pts = torch.as_tensor(rng.uniform(0, 1, (64, 3)), **dev)
        R = _rotations(rng.uniform(0, 1, (64, 3)))
        M = R @ np.diag([1.0, 1e-3, 1e-3]) @ R.transpose(0, 2, 1)
        M = torch.as_tensor(np.stack([M[:, 0, 0], M[:, 1, 1], M[:, 2, 2], M[:, 0, 1], M[:, 0, 2], M[:, 1, 2]]), **dev)
        cz, cy, cx = ((torch.arange(q, **dev) + 0.5) / q for q in (nz, ny, nx))
        best = torch.full((nz, ny, nx), 1e30, **dev)
        reg = torch.zeros((nz, ny, nx), device="cuda", dtype=torch.int64)
        for k in range(64):
            d = (cz - pts[k, 2])[:, None, None] ** 2 + (cy - pts[k, 1])[None, :, None] ** 2 + (cx - pts[k, 0]) ** 2
            m = d < best
            best = torch.where(m, d, best)
            reg = torch.where(m, torch.full_like(reg, k), reg)
        K = M[:, reg.reshape(-1)].reshape(6, nz, ny, nx).contiguous()
    else:  # inclusions: spheres of 1e6 in diag(1, 1, 1e-2), a fifth of the volume
        inside = torch.zeros((nz, ny, nx), device="cuda", dtype=torch.bool)
        vol = 0.0
        z, y, x = (torch.arange(q, **dev) + 0.5 for q in (nz, ny, nx))
        while vol < 0.23 * nx * ny * nz:
            c, r = rng.uniform(0, 1, 3) * (nx, ny, nz), rng.uniform(4.0, 12.0)
            lo = [max(0, int(v - r) - 1) for v in c]
            hi = [min(q, int(v + r) + 2) for v, q in zip(c, (nx, ny, nz))]
            sx, sy, sz = (slice(a, b) for a, b in zip(lo, hi))
            d = (z[sz] - c[2])[:, None, None] ** 2 + (y[sy] - c[1])[None, :, None] ** 2 + (x[sx] - c[0]) ** 2
            inside[sz, sy, sx] |= d < r * r
            vol += 4.0 / 3.0 * math.pi * r ** 3
        for c, base in enumerate((1.0, 1.0, 1e-2)):
            K[c] = torch.where(inside, 1e6, base)
    return K


def _element(dim, h):
    """Symmetric 2^dim x 2^dim matrices of the packed components (xx, yy[, zz, xy, xz, yz] / xy) on one box element."""
    M, S, C = [], [], []
    for a in range(dim):
        M.append(h[a] / 6 * np.array([[2.0, 1.0], [1.0, 2.0]]))
        S.append(np.array([[1.0, -1.0], [-1.0, 1.0]]) / h[a])
        C.append(0.5 * np.array([[-1.0, -1.0], [1.0, 1.0]]))   # int phi_i' phi_j
    pairs = [(a, a) for a in range(dim)] + ([(0, 1), (0, 2), (1, 2)] if dim == 3 else [(0, 1)])
    out = []
    for a, b in pairs:
        G = np.zeros((1 << dim, 1 << dim))
        for i in range(1 << dim):
            for j in range(1 << dim):
                v = 1.0
                for c in range(dim):
                    ic, jc = (i >> c) & 1, (j >> c) & 1
                    if a == b:
                        v *= S[c][ic, jc] if c == a else M[c][ic, jc]
                    else:
                        v *= C[c][ic, jc] if c == a else (C[c][jc, ic] if c == b else M[c][ic, jc])
                G[i, j] = v
        out.append(0.5 * (G + G.T) if a == b else G + G.T)
    return out


def _operator(case, seed, gi=0):
    """The problem dict of sa.Hierarchy, on the device."""
    rng = np.random.RandomState((seed * 7919 + 104729 * gi) % (1 << 31))
    (nx, ny, nz), h = _grid(case, gi)
    dim = 3 if nz else 2
    K = _tensors(case, (nx, ny, nz), rng, gi)
    nzz = max(nz, 1)
    Nx, Ny, Nz = nx + 1, ny + 1, nz + 1
    n = Nx * Ny * Nz
    G = _element(dim, h)
    noff = 3 ** dim
    V = torch.zeros((noff, Nz, Ny, Nx), device="cuda", dtype=torch.float64)
    for i in range(1 << dim):
        at = [(i >> c) & 1 for c in range(3)]
        sl = (slice(at[2], at[2] + nzz), slice(at[1], at[1] + ny), slice(at[0], at[0] + nx))
        for j in range(1 << dim):
            o = [((j >> c) & 1) - at[c] for c in range(dim)]
            off = sum((o[c] + 1) * 3 ** c for c in range(dim))
            acc = None
            for c, g in enumerate(G):
                if g[i, j] != 0.0 and (case["kind"] == "voronoi" or c < dim):
                    acc = K[c] * g[i, j] if acc is None else acc + K[c] * g[i, j]
            V[(off,) + sl] += acc
    # Dirichlet nodes: x = 0 (battery: bottom and top, two_domain: the whole boundary); their columns are eliminated
    free = torch.ones((Nz, Ny, Nx), device="cuda", dtype=torch.bool)
    if case["kind"] == "battery":
        free[0], free[-1] = False, False
    else:
        free[:, :, 0] = False
        if case["kind"] == "two_domain":
            free[:, :, -1], free[:, 0], free[:, -1] = False, False, False
    pad = torch.zeros((Nz + 2, Ny + 2, Nx + 2), device="cuda", dtype=torch.bool)
    pad[1:-1, 1:-1, 1:-1] = free
    keep = torch.zeros((noff, Nz, Ny, Nx), device="cuda", dtype=torch.bool)
    step = torch.zeros(noff, device="cuda", dtype=torch.int64)
    for off in range(noff):
        ox, oy, oz = off % 3 - 1, (off // 3) % 3 - 1, off // 9 - 1 if dim == 3 else 0
        keep[off] = free & pad[1 + oz:1 + oz + Nz, 1 + oy:1 + oy + Ny, 1 + ox:1 + ox + Nx]
        step[off] = ox + Nx * (oy + Ny * oz)
    keep[noff // 2] = True
    V[noff // 2][~free] = 1.0   # a Dirichlet row holds only its diagonal
    keep = keep.reshape(noff, n).t()
    V = V.reshape(noff, n).t()
    cnt = keep.sum(1)
    rp = torch.zeros(n + 1, device="cuda", dtype=torch.int64)
    torch.cumsum(cnt, 0, out=rp[1:])
    val = V[keep]
    col = (torch.arange(n, device="cuda", dtype=torch.int32)[:, None] + step.to(torch.int32)[None, :])[keep]
    del V, keep
    X = torch.meshgrid(*(torch.arange(q, device="cuda", dtype=torch.float64) * s
                         for q, s in zip((Nz, Ny, Nx), (h[2], h[1], h[0]))), indexing="ij")
    coords = torch.stack([X[2], X[1], X[0]][:dim], -1).reshape(-1).contiguous()
    e = torch.meshgrid(*(torch.arange(q, device="cuda", dtype=torch.int64) for q in (nzz, ny, nx)), indexing="ij")
    base = (e[2] + Nx * (e[1] + Ny * e[0])).reshape(-1)
    nodes = torch.stack([base + (l & 1) + Nx * (((l >> 1) & 1) + Ny * (l >> 2)) for l in range(1 << dim)], 1)
    ne = base.numel()
    return dict(dim=dim, n=n, nnz=int(rp[-1]), row_ptr=rp, col=col, val=val, coords=coords, tloc="element",
                tensors=K.reshape(K.shape[0], -1).t().contiguous().reshape(-1),
                elem_nodes=nodes.to(torch.int32).reshape(-1).contiguous(),
                elem_measure=torch.full((ne,), float(np.prod(h[:dim])), device="cuda", dtype=torch.float64)), free.reshape(-1)


def _rhs(seed, k, free):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 31 + 7)
    return torch.randn((k, free.numel()), generator=g, device="cuda", dtype=torch.float64) * free


def _setup(case, p):
    return sa.Hierarchy(p, theta=THETA[case["measure"]], measure=case["measure"], precision=case["precision"],
                        max_coarse=case["max_coarse"])


def prepare(case, seed):
    op = case["op"]
    if op == "group":
        hs, bs = [], []
        for gi in range(case["m"]):
            p, free = _operator(case, seed, gi)
            hs.append(_setup(case, p))
            bs.append(_rhs(seed + gi, 1, free)[0])
        return dict(case=case, h=hs, b=bs)
    p, free = _operator(case, seed)
    if op == "strength":
        # what a caller of the filter holds: the matrix, the nodal inverse tensors, the Dirichlet flags
        st = dict(case=case, p=p, dirichlet=(~free).to(torch.uint8))
        kp = 6
        sig = torch.zeros((p["n"], kp), device="cuda", dtype=torch.float64)
        w = torch.zeros(p["n"], device="cuda", dtype=torch.float64)
        en, t = p["elem_nodes"].reshape(-1, 8).long(), p["tensors"].reshape(-1, kp)
        ex, ey, ez = _grid(case)[0]
        tg, sg, wg = t.reshape(ez, ey, ex, kp), sig.reshape(ez + 1, ey + 1, ex + 1, kp), w.reshape(ez + 1, ey + 1, ex + 1)
        for l in range(8):
            s = (slice(l >> 2, (l >> 2) + ez), slice((l >> 1) & 1, ((l >> 1) & 1) + ey), slice(l & 1, (l & 1) + ex))
            sg[s] += tg
            wg[s] += 1.0
        del en
        a, b, c, d, e, f = (sig / w[:, None]).unbind(1)   # xx yy zz xy xz yz
        det = a * (b * c - f * f) - d * (d * c - f * e) + e * (d * f - b * e)
        inv = torch.stack([b * c - f * f, a * c - e * e, a * b - d * d, e * f - d * c, d * f - b * e, d * e - a * f], 1)
        st["sinv"] = (inv / det[:, None]).contiguous()
        return st
    st = dict(case=case, p=p)
    B = _rhs(seed, case.get("k", 1), free)
    st["b"] = B if op == "batch" else B[0]
    if op in ("solve", "batch"):
        st["h"] = _setup(case, p)
        del st["p"]
    return st


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "solve":
        x, info = state["h"].solve(state["b"], tol=TOL)
        return dict(x=x, iters=info["iters"])
    if op == "batch":
        X, infos = state["h"].solve_batch(state["b"], tol=TOL)
        return dict(x=X, iters=[i["iters"] for i in infos])
    if op == "group":
        X, infos = sa.solve_group(state["h"], state["b"], tol=TOL)
        return dict(x=X, iters=[i["iters"] for i in infos])
    if op == "strength":
        p = state["p"]
        return sa.strength(case["measure"], 3, p["row_ptr"], p["col"], p["val"], p["coords"], state["sinv"],
                           state["dirichlet"], THETA[case["measure"]])
    h = _setup(case, state["p"])
    if op == "setup_apply":
        out = h.vcycle(state["b"])
    else:
        x, info = h.solve(state["b"], tol=TOL)
        out = dict(x=x, iters=info["iters"])
    h.free()
    return out


def _size(case, gi=0):
    (nx, ny, nz), _ = _grid(case, gi)
    n = (nx + 1) * (ny + 1) * (nz + 1)
    return n, n * (27 if nz else 9)


def work(case):
    """What a pass cannot do without: per V-cycle and CG iteration five products with the fine operator (two
    smoothing steps that need one before the coarse correction's residual, the residual, two after, one of CG),
    each reading every stored entry (value and column) and the vectors it combines; setup: the matrix read by the
    strength measure, the filter, the two Galerkin products and written once for the solve.  Coarse levels, which
    hold a fraction of the entries, are left out."""
    op = case["op"]
    by = fl = 0.0
    for gi in range(case["m"] if op == "group" else 1):
        n, nnz = _size(case, gi)
        k = case.get("k", 1)
        v = 4 if case.get("precision") == "fp32" else 8
        if op == "strength":
            by += 12 * nnz + (9 * 8) * n + nnz
            fl += 40 * nnz / 2 if case["measure"] == "material" else 3 * nnz
            continue
        its = 1 if op == "setup_apply" else CYCLES[case["kind"]]
        by += its * (4 * ((v + 2) * nnz + 4 * v * n * k) + (10 * nnz + 24 * n * k if op != "setup_apply" else 0))
        fl += its * k * 10 * nnz
        if op in ("setup_solve", "setup_apply"):
            by += 4 * 12 * nnz + (v + 2) * nnz
            fl += 30 * nnz
    return dict(bytes=float(by), flops=float(fl))


# ---------------------------------------------------------------------------
# the solution in 64 bits by plain torch: a dense solve of the small systems, Jacobi-preconditioned CG run far below
# TOL on those up to about 1e6 unknowns; the strength mask and the V-cycle have no value of their own here
# ---------------------------------------------------------------------------
def _plain_solve(p, b):
    n = p["n"]
    A = torch.sparse_csr_tensor(p["row_ptr"], p["col"].long(), p["val"], (n, n))
    if n <= 6000:
        return torch.linalg.solve(A.to_dense(), b)
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), p["row_ptr"].diff())
    d = p["val"][row == p["col"]]
    x = torch.zeros_like(b)
    r = b.clone()
    z = r / d
    q = z.clone()
    rz = r @ z
    goal = float(b.norm()) * 1e-12
    for it in range(12000):
        Aq = A @ q
        a = rz / (q @ Aq)
        x += a * q
        r -= a * Aq
        if it % 50 == 49 and float(r.norm()) < goal:
            return x
        z = r / d
        new = r @ z
        q = z + (new / rz) * q
        rz = new
    return None


def exact(case, seed):
    op = case["op"]
    if op == "group":
        out = []
        for gi in range(case["m"]):
            p, free = _operator(case, seed, gi)
            out.append(_plain_solve(p, _rhs(seed + gi, 1, free)[0]) if p["n"] <= 6000 else None)
        return dict(x=out, iters=None)
    if op not in ("solve", "setup_solve") or _size(case)[0] > 1.2e6 or case["kind"] == "inclusions":
        return None
    p, free = _operator(case, seed)
    x = _plain_solve(p, _rhs(seed, 1, free)[0])
    return None if x is None else dict(x=x, iters=None)
