"""CUDA kernels at the sizes where their tiling can go wrong: the coarse factor
and solve around tiles of 32 rows and diagonal blocks of 1024, the CG
reductions around a block of 256 rows and the full grid, SpGEMM rows around
its tiers, and the strength masks around 64-row blocks, ties and extreme
exponents."""
import numpy as np
import pytest
import scipy.sparse as sp
from test_gpu_parity import compare

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


@pytest.fixture(scope="module")
def sa():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2602_05686_gb300 as m
    m.build()
    return m


def problem(A, dim=2, coords=None):
    A = sp.csr_matrix(A)
    A.sort_indices()
    n = A.shape[0]
    if coords is None:
        coords = np.stack([np.arange(n)] + [np.zeros(n)] * (dim - 1), 1).astype(np.float64)
    iso = [1.0, 0.0, 1.0] if dim == 2 else [1.0, 0.0, 0.0, 1.0, 0.0, 1.0]
    return dict(dim=dim, n=n, nnz=A.nnz, row_ptr=A.indptr.astype(np.int64), col=A.indices.astype(np.int32),
                val=A.data.astype(np.float64), coords=coords.ravel(), tloc="node", tensors=np.tile(iso, n))


def laplacian(n, i, j, w, shift):
    """weighted graph Laplacian + shift"""
    W = sp.coo_matrix((w, (i, j)), shape=(n, n)).tocsr()
    W = W + W.T
    return sp.csr_matrix(sp.diags(np.asarray(W.sum(1)).ravel() + shift) - W)


def coarse_matrix(n, pattern, rng):
    i = np.arange(n - 1)
    if pattern == "blocks":  # components of 100 rows: tiles outside the skyline between them
        i = i[(i + 1) % 100 != 0]
        i, j = np.concatenate([i, i[i % 100 < 60]]), np.concatenate([i + 1, i[i % 100 < 60] + 39])
        j = np.minimum(j, n - 1)
    elif pattern == "band":
        i, j = np.concatenate([i, i[:max(n - 40, 0)]]), np.concatenate([i + 1, i[:max(n - 40, 0)] + 40])
    else:  # scattered: the skyline reaches the first tiles from every tile row
        j = np.concatenate([i + 1, rng.integers(0, n, 3 * n)])
        i = np.concatenate([i, rng.integers(0, n, 3 * n)])
    m = i != j
    return laplacian(n, i[m], j[m], 0.5 + rng.random(m.sum()), 0.5)


@pytest.mark.parametrize("pattern", ["band", "blocks", "scattered"])
@pytest.mark.parametrize("n", [2, 31, 32, 33, 64, 65, 1023, 1024, 1025, 2049, 3000])
def test_coarse_factor_and_solve(sa, n, pattern):
    """one-level hierarchy = the coarse direct solve.  Bar: the normwise residual
    bound of Cholesky, 3 n eps |L||L^T| <= 3 n eps * 2 |A| for a diagonally
    dominant A, with a factor for the inverted diagonal blocks: 16 n eps
    |A| |z|."""
    import torch
    rng = np.random.default_rng(n)
    A = coarse_matrix(n, pattern, rng)
    h = sa.Hierarchy(problem(A), measure="material", max_coarse=5000)
    assert h.stats()["levels"] == 1
    B = rng.standard_normal((3, n))
    Bd = torch.from_numpy(B).cuda()
    z = h.vcycle(Bd[0].contiguous()).cpu().numpy()
    res = np.abs(B[0] - A @ z).max()
    assert res <= 16 * n * EPS * abs(A).sum(1).max() * np.abs(z).max()
    X, infos = h.solve_batch(Bd)
    h2 = sa.Hierarchy(problem(coarse_matrix(33, "band", rng)), measure="material", max_coarse=5000)
    b2 = torch.from_numpy(rng.standard_normal(33)).cuda()
    G, _ = sa.solve_group([h, h2], [Bd[0].contiguous(), b2])
    for c in range(3):
        x1, i1 = h.solve(Bd[c].contiguous())
        assert infos[c]["iters"] == i1["iters"] and torch.equal(X[c], x1)
        if c == 0:
            assert torch.equal(G[0], x1)
    assert torch.equal(G[1], h2.solve(b2)[0])


@pytest.mark.parametrize("n", [33, 1025])
def test_coarse_factor_reports_a_late_bad_pivot(sa, n):
    A = coarse_matrix(n, "band", np.random.default_rng(1)).tolil()
    w = 2.0 * np.sqrt(A[n - 1, n - 1] * A[n - 2, n - 2])
    A[n - 1, n - 2] = A[n - 2, n - 1] = -w
    with pytest.raises(sa.SAError) as e:
        sa.Hierarchy(problem(A), measure="material", max_coarse=5000)
    assert e.value.status == -4


@pytest.mark.parametrize("n", [255, 256, 257, 271, 272, 273, 511, 512, 513, 304 * 512 - 1, 304 * 512, 304 * 512 + 1,
                               4096 * 256 - 1, 4096 * 256 + 1])
def test_reductions_at_block_and_grid_edges(sa, n):
    """the reported residual norm against numpy's.  Bar: both sides form b - A x
    with at most 4 roundings per entry of |b| + |A||x| and sum n squares in
    trees or in order; 16 eps (|b| + |A||x|) in norm covers the residual and
    n eps relative the sum."""
    import torch
    e = np.ones(n - 1)
    A = sp.csr_matrix(sp.diags([-e, np.full(n, 2.05), -e], [-1, 0, 1]))
    h = sa.Hierarchy(problem(A), theta=0.08, measure="material", max_coarse=64)
    k = 5 if n < 10 ** 6 else 2  # blocks of eight (two lanes a row) and of two columns
    B = np.random.default_rng(n).standard_normal((k, n))
    Bd = torch.from_numpy(B).cuda()
    X, infos = h.solve_batch(Bd)
    for c in range(k):
        x, i = h.solve(Bd[c].contiguous())
        assert i["status"] == 0 and i["iters"] == infos[c]["iters"] and torch.equal(x, X[c])
        x = x.cpu().numpy()
        nb = np.linalg.norm(B[c])
        ref = np.linalg.norm(B[c] - A @ x) / nb
        slack = 16 * EPS * np.linalg.norm(np.abs(B[c]) + abs(A) @ np.abs(x)) / nb
        assert i["rel_res"] <= 1e-8
        assert abs(i["rel_res"] - ref) <= slack + n * EPS * ref


@pytest.mark.parametrize("passes", ["1", "2"])
@pytest.mark.parametrize("size", [4, 40])
def test_spgemm_rows_at_the_tier_edges(sa, orc, monkeypatch, passes, size):
    """cliques of `size` rows (one aggregate each) and hub rows coupled weakly to
    d of them: the hub's row of A P has exactly d + 1 columns (24: the thread
    tier's lists, 32: a warp's round, 192: the warp tier's table), diagonal-only
    rows have none.  64 rows of the larger cliques hold more entries than the
    filter stages."""
    nc, hubs = 450, [1, 22, 23, 24, 30, 31, 32, 190, 191, 192, 193, 400]
    a, b = np.triu_indices(size, 1)
    i = (np.arange(nc)[:, None] * size + a).ravel()
    j = (np.arange(nc)[:, None] * size + b).ravel()
    w = np.ones(i.size)
    for k, d in enumerate(hubs):
        hub = (nc - 1 - k) * size
        t = np.arange(d) * size + size // 2
        i, j, w = np.concatenate([i, np.full(d, hub)]), np.concatenate([j, t]), np.concatenate([w, np.full(d, 1e-3)])
    n = nc * size + 3
    p = problem(laplacian(n, i, j, w, 0.1))
    monkeypatch.setenv("SA_SPGEMM_PASSES", passes)
    h = sa.Hierarchy(p, theta=0.01, measure="classical", max_coarse=50, max_levels=2, keep_setup_data=True)
    o = orc.Hierarchy(p, 0.01, "classical", max_coarse=50, max_levels=2)
    assert o.nlev == 2 and o.level(1)["n"] == nc
    compare(h, o, orc=orc)


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("n", [2, 63, 64, 65, 129, 1000])
@pytest.mark.parametrize("kind", ["symmetric", "pattern", "scales", "lattice"])
def test_strength_masks(sa, orc, dim, n, kind):
    """bit for bit the oracle's: a symmetric pattern, one that is not, tensors
    whose products leave the FP32 comparison's exponents, and lattice points with
    equal tensors (ties); classical with entries of both signs and ties"""
    import torch
    rng = np.random.default_rng(100 * dim + n)
    P = sp.random(n, n, min(1.0, 12.0 / n), random_state=rng, format="csr") + sp.eye(n)
    if kind != "pattern":
        P = P + P.T
    P = sp.csr_matrix(P)
    P.sort_indices()
    rp, ci = P.indptr.astype(np.int64), P.indices.astype(np.int32)
    if kind == "lattice":
        x = np.stack(np.unravel_index(rng.permutation(4096)[:n], (16, 16, 16)), 1)[:, :dim].astype(np.float64)
        x[:, 0] += 16.0 * np.arange(n)  # distinct points
    else:
        x = rng.random((n, dim))
    kp = 3 if dim == 2 else 6
    few = np.zeros((4, kp))
    few[:, [0, 2] if dim == 2 else [0, 3, 5]] = 1.0 + rng.random((4, dim))
    few[:, 1] = 0.3
    s = few[rng.integers(0, 1 if kind == "lattice" else 4, n)]
    if kind == "scales":
        s = s * 10.0 ** rng.choice([-140.0, -60.0, 0.0, 60.0, 140.0], n)[:, None]
    dirm = (rng.random(n) < 0.05).astype(np.uint8)
    v = rng.choice([-1.0, -0.5, -0.25, 0.25, 0.5], ci.size)
    v[ci == np.repeat(np.arange(n), np.diff(rp))] = 1.0
    if kind == "scales":
        v = v * 10.0 ** rng.choice([-150.0, 0.0, 150.0], ci.size)
    t = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)  # noqa: E731
    g = [t(rp, torch.int64), t(ci, torch.int32), t(v, torch.float64), t(x.ravel(), torch.float64),
         t(s.ravel(), torch.float64), t(dirm, torch.uint8)]
    for theta in (0.0, 0.05, 0.25, 0.5):
        _, _, ko = orc.strength_material(dim, n, rp, ci, dirm, x, s, theta)
        kg = sa.strength("material", dim, g[0], g[1], None, g[3], g[4], g[5], theta)
        assert np.array_equal(kg.cpu().numpy(), ko), theta
        kc = sa.strength("classical", dim, g[0], g[1], g[2], None, None, g[5], theta)
        assert np.array_equal(kc.cpu().numpy(), orc.strength_classical(n, rp, ci, v, dirm, theta)), theta


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("kind", ["all", "one", "descending", "duplicates"])
@pytest.mark.parametrize("n", [3, 64, 65, 1000])
def test_strength_of_rows_in_any_order(sa, orc, dim, n, kind):
    """sa_strength asks for no order of a row's columns: bit for bit the oracle's
    mask, which takes the entries as they stand; every row shuffled, one row of
    one 64-row block, descending rows, repeated columns"""
    import torch
    rng = np.random.default_rng(7 * dim + n)
    P = sp.random(n, n, min(1.0, 20.0 / n), random_state=rng, format="csr") + sp.eye(n)
    P = sp.csr_matrix(P + P.T)
    P[n // 2, :min(n, 50)] = 1.0  # a row of more than a warp's lanes
    P = sp.csr_matrix(P)
    P.sort_indices()
    rp, ci = P.indptr.astype(np.int64), P.indices.astype(np.int32)
    v = rng.choice([-1.0, -0.5, 0.25], ci.size)
    rows = [n // 2] if kind == "one" else range(n)
    for i in rows:
        b, e = rp[i], rp[i + 1]
        o = np.arange(e - b)[::-1] if kind == "descending" else rng.permutation(e - b)
        ci[b:e] = ci[b:e][o]
        if kind == "duplicates" and e - b > 2:
            ci[b + 1] = ci[b]
    x = rng.random((n, dim))
    kp = 3 if dim == 2 else 6
    s = np.zeros((n, kp))
    s[:, :dim] = 1.0 + rng.random((n, dim))
    s[:, dim] = 0.2
    dirm = (rng.random(n) < 0.05).astype(np.uint8)
    t = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)  # noqa: E731
    g = [t(rp, torch.int64), t(ci, torch.int32), t(v, torch.float64), t(x.ravel(), torch.float64),
         t(s.ravel(), torch.float64), t(dirm, torch.uint8)]
    iso = np.zeros((n, kp))
    iso[:, :dim] = 1.0
    for theta in (0.05, 0.3):
        _, _, ko = orc.strength_material(dim, n, rp, ci, dirm, x, s, theta)
        kg = sa.strength("material", dim, g[0], g[1], None, g[3], g[4], g[5], theta)
        assert np.array_equal(kg.cpu().numpy(), ko), theta
        _, _, ko = orc.strength_material(dim, n, rp, ci, dirm, x, iso, theta)
        kg = sa.strength("distance", dim, g[0], g[1], None, g[3], None, g[5], theta)
        assert np.array_equal(kg.cpu().numpy(), ko), theta
        if kind != "duplicates":  # (a repeated diagonal: which of them is the diagonal is not defined)
            kc = sa.strength("classical", dim, g[0], g[1], g[2], None, None, g[5], theta)
            assert np.array_equal(kc.cpu().numpy(), orc.strength_classical(n, rp, ci, v, dirm, theta)), theta


def test_spgemm_scratch_that_cannot_be_had(sa, gen_mod, monkeypatch):
    """an allocator that has the memory of the two-phase products but not the
    one-pass form's scratch: setup falls back and gives the same hierarchy, bit
    for bit"""
    import ctypes
    import torch
    p = gen_mod.battery_3d(12, 12, 24)
    t = {k: torch.from_numpy(np.ascontiguousarray(p[k])).cuda() for k in ("row_ptr", "col", "val", "coords")}
    b = np.random.default_rng(5).standard_normal(p["n"])
    b[p["dir_mask"] == 1] = 0.0
    bd = torch.from_numpy(b).cuda()
    L = sa.lib()

    def run(limit):
        live, most, refused = {}, [0], [0]

        @sa.api._ALLOC
        def alloc(nbytes, ctx):
            if nbytes > limit:
                refused[0] += 1
                return None
            most[0] = max(most[0], int(nbytes))
            buf = torch.empty(int(nbytes) + 256, dtype=torch.uint8, device="cuda")
            ptr = (buf.data_ptr() + 255) // 256 * 256
            live[ptr] = buf
            return ptr

        @sa.api._FREE
        def free(ptr, ctx):
            live.pop(ptr, None)

        o = sa.default_options()
        o.max_coarse, o.measure = 100, 0
        o.stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        o.alloc, o.dealloc = alloc, free
        pr = sa.Problem()
        pr.dim, pr.n, pr.nnz = 3, p["n"], p["nnz"]
        pr.row_ptr, pr.col, pr.val = t["row_ptr"].data_ptr(), t["col"].data_ptr(), t["val"].data_ptr()
        pr.coords = t["coords"].data_ptr()
        hh = ctypes.c_void_p()
        assert L.sa_setup(ctypes.byref(pr), ctypes.byref(o), ctypes.byref(hh)) == 0
        x = torch.zeros_like(bd)
        info = sa.SolveInfo()
        assert L.sa_solve(hh, bd.data_ptr(), x.data_ptr(), 1e-8, ctypes.byref(info)) == 0
        torch.cuda.synchronize()
        L.sa_free(hh)
        assert not live
        return x.cpu(), info.iters, most[0], refused[0]

    one = run(1 << 40)
    monkeypatch.setenv("SA_SPGEMM_PASSES", "2")
    two = run(1 << 40)
    monkeypatch.delenv("SA_SPGEMM_PASSES")
    assert one[2] > two[2]  # the scratch is the largest request
    none = run(two[2])
    assert none[3] > 0
    for r in (two, none):
        assert torch.equal(one[0], r[0]) and one[1] == r[1]


@pytest.mark.parametrize("n", [100, 1100])
def test_coarse_solve_bytes_are_the_entries_it_reads(sa, n):
    """the profile's algorithmic bytes of a coarse solve: the diagonal blocks'
    triangles twice, and of the rows between blocks the tiles inside the skyline
    (bandwidth 40: two tile rows reach back 64 and 32 columns, two tile columns
    forward 32 and 64)"""
    import torch
    A = coarse_matrix(n, "band", np.random.default_rng(1))
    h = sa.Hierarchy(problem(A), measure="material", max_coarse=5000)
    b = torch.from_numpy(np.random.default_rng(2).standard_normal(n)).cuda()
    sa.profile_enable(True)
    h.vcycle(b)
    rows = [r for r in sa.profile_read() if r["kind"] == "coarse"]
    sa.profile_enable(False)
    tri = n * (n + 1) if n <= 1024 else 1024 * 1025 + (n - 1024) * (n - 1023)
    between = 0 if n <= 1024 else 2 * (32 * 64 + 32 * 32)
    assert len(rows) == 1 and rows[0]["launches"] == 1
    assert rows[0]["bytes"] == 8.0 * (tri + between) + 32.0 * n


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("n", [25, 32, 33, 161, 200])
@pytest.mark.parametrize("order", ["ascending", "any"])
def test_strength_of_few_long_rows(sa, orc, dim, n, order):
    """small levels of long rows (a warp per row, blocks of eight rows): dense and
    half-dense rows of 25 to 200 entries, bit for bit the oracle's masks"""
    import torch
    rng = np.random.default_rng(11 * dim + n)
    for density in (1.0, 0.6 if n > 60 else 1.0):
        P = sp.csr_matrix((rng.random((n, n)) < density) | np.eye(n, dtype=bool))
        P = sp.csr_matrix(P + P.T)
        P.sort_indices()
        rp, ci = P.indptr.astype(np.int64), P.indices.astype(np.int32)
        assert ci.size > 24 * n
        if order == "any":
            for i in range(n):
                ci[rp[i]:rp[i + 1]] = rng.permutation(ci[rp[i]:rp[i + 1]])
        v = rng.choice([-1.0, -0.5, 0.25, 0.0, -0.0], ci.size)
        v[ci == np.repeat(np.arange(n), np.diff(rp))] = rng.choice([1.0, -1.0], n)
        x = rng.random((n, dim))
        kp = 3 if dim == 2 else 6
        s = np.zeros((n, kp))
        s[:, :dim] = 1.0 + rng.integers(0, 3, (n, dim))
        dirm = (rng.random(n) < 0.05).astype(np.uint8)
        t = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)  # noqa: E731
        g = [t(rp, torch.int64), t(ci, torch.int32), t(v, torch.float64), t(x.ravel(), torch.float64),
             t(s.ravel(), torch.float64), t(dirm, torch.uint8)]
        for theta in (0.0, 0.01, 0.25):
            _, _, ko = orc.strength_material(dim, n, rp, ci, dirm, x, s, theta)
            kg = sa.strength("material", dim, g[0], g[1], None, g[3], g[4], g[5], theta)
            assert np.array_equal(kg.cpu().numpy(), ko), theta
            kc = sa.strength("classical", dim, g[0], g[1], g[2], None, None, g[5], theta)
            assert np.array_equal(kc.cpu().numpy(), orc.strength_classical(n, rp, ci, v, dirm, theta)), theta
