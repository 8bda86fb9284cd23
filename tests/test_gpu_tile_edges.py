"""Kernels at the edges of their tiles: remainders, the smallest sizes, ragged rows, against the
FP64 oracle or the definition.  Tolerances are derived beside each test."""
import numpy as np
import pytest

from oracle import learned as L

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


# n * m entries: one, just below / at / above a tile of 128, one tile a CTA over the whole grid
# (3 x 152 tiles) and a ragged tile more
@pytest.mark.parametrize("n,m", [(1, 1), (127, 1), (16, 8), (43, 3), (456 * 16, 8), (19457, 3)])
def test_lp_grad_tile_edges(n, m):
    from paper_2305_15552_gb300 import binding as B
    rng = np.random.default_rng(n + m)
    F = rng.standard_normal((n, m, 6)) * [60, 1, 60, 60, 1, 10] + [150, 1, 150, 170, 0, 0]
    F = F.astype(np.float32)
    r = (1e-2 * rng.standard_normal((n, m))).astype(np.float32)
    z = (r / 50 * (1 + 0.3 * rng.standard_normal((n, m)))).astype(np.float32)
    colw = 1.0 / (m * (z.astype(np.float64) ** 2).sum(0))
    p = (0.3 * rng.standard_normal(L.N_PARAMS)).astype(np.float32)
    p[:12] = [150, 1, 150, 170, 0, 0, 60, 1, 60, 60, 1, 10]
    s = dict(F=_dev(F.reshape(-1, 6)), r=_dev(r.reshape(-1)), z=_dev(z.reshape(-1)), colw=_dev(colw), n=n, m=m)
    g = B.lp_grad(_dev(p), s).cpu().numpy()
    Lo, go = L.loss_grad(p.astype(np.float64), F.astype(np.float64), r.astype(np.float64), z.astype(np.float64),
                         colw * m)
    # FP32 chains of 6 + 32 + 32 + 128 products: a normwise error of ~200 * 2^-24 = 1.2e-5 at worst,
    # and the loss sums squares of differences that keep two to three digits of z
    assert g[-1] == pytest.approx(Lo, rel=1e-4)
    gt = go[L.N_FIXED:]
    for a, b in [(12, 204), (204, 236), (236, 1260), (1260, 1292), (1292, 1324), (1324, 1325)]:
        ga, gb = g[a - 12:b - 12], gt[a - 12:b - 12]
        assert np.linalg.norm(ga - gb) <= 1e-4 * max(np.linalg.norm(gb), 1e-2 * np.linalg.norm(gt)), (a, b)


def _shifted(a, dt):
    """The array on the device one element past a 16-byte boundary."""
    flat = torch.empty(a.size + 1, dtype=dt, device="cuda")
    v = flat[1:].view(a.shape)
    v.copy_(torch.tensor(a, dtype=dt))
    return v


# rows: one, around a chunk of 32, one chunk a CTA (304 CTAs), several chunk groups a CTA with a
# ragged last one; widths with 1 x 1, 2 x 2, 4 x 4 tiles, and more tiles than threads
@pytest.mark.parametrize("n", [1, 31, 33, 304 * 32, 304 * 32 * 3 + 45, 200003])
@pytest.mark.parametrize("nb", [5, 6, 8, 16, 64])
@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
def test_gram_chunk_edges(n, nb, dt):
    from paper_2305_15552_gb300 import binding as B
    rng = np.random.default_rng(n + nb)
    a, b = rng.standard_normal((n, nb)), rng.standard_normal((n, nb))
    A, Bm = torch.tensor(a, dtype=dt, device="cuda"), torch.tensor(b, dtype=dt, device="cuda")
    for X, Y in ((A, Bm), (A, A), (_shifted(a, dt), Bm)):
        G = B.gram(X, Y).cpu().numpy()
        Xe, Ye = X.double().cpu().numpy(), Y.double().cpu().numpy()
        bound = np.abs(Xe).T @ np.abs(Ye)
        # FP32: products rounded once and summed over 32 rows (at most 33 * 2^-24 of the sum of
        # magnitudes), the rest exact to 2^-40; FP64: n terms of 2^-53
        tol = (2.0 ** -24 * 40 if dt == torch.float32 else 2.0 ** -53 * (n + 10)) * bound + 1e-300
        assert np.all(np.abs(G - Xe.T @ Ye) <= tol)
        if X is Y:
            assert np.array_equal(G, G.T)


# rows: fewer than one warp pass, around the 256 / 512 rows of a CTA pass, ragged; widths with the
# in-place apply (8, 16) and without; a block off the 16-byte boundary
@pytest.mark.parametrize("n", [16, 31, 257, 1025, 608 * 512 + 7])
@pytest.mark.parametrize("k", [5, 8, 16])
@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
@pytest.mark.parametrize("shift", [False, True])
def test_cholqr2_row_edges(n, k, dt, shift):
    from paper_2305_15552_gb300 import binding as B
    x = np.random.default_rng(n + k).standard_normal((n, k)) * np.logspace(0, -1, k)
    X = _shifted(x, dt) if shift else torch.tensor(x, dtype=dt, device="cuda")
    Xe = X.double().cpu().numpy()
    Q, R = B.cholqr2(X)
    Q, R = Q.double().cpu().numpy(), R.cpu().numpy()
    eps = 2.0 ** -24 if dt == torch.float32 else 2.0 ** -53
    # the second pass works on a basis orthonormal to ~cond^2 eps: Q^T Q - I is a few rounding errors
    # of k-term rows and of the Gram; Q R reproduces X to two k-term products per pass
    assert np.abs(Q.T @ Q - np.eye(k)).max() < 40 * k * eps
    assert np.abs(Q @ R - Xe).max() < 40 * k * eps * np.abs(Xe).max()
    assert np.array_equal(R, np.triu(R))


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
def test_cholqr2_breakdown_leaves_block(dt):
    from paper_2305_15552_gb300 import binding as B
    x = np.random.default_rng(3).standard_normal((3000, 8))
    x[:, 5] = 0.0                        # a pivot of exactly zero
    X = torch.tensor(x, dtype=dt, device="cuda")
    Y = X.clone()
    with pytest.raises(B.EigError) as e:
        B.cholqr2(X)
    assert e.value.status == B.EIG_EBREAKDOWN
    assert torch.equal(X, Y)


# row blocks: one fewer and one more than the 152 SMs' worth at which a row block stops being split
# into two CTAs (the last one ragged), and a single row block of a few rows
@pytest.mark.parametrize("n", [40, 151 * 256 + 9, 152 * 256 + 9])
@pytest.mark.parametrize("val,dt,nb", [("f32", torch.float32, 1), ("f32", torch.float32, 16), ("f32", torch.float64, 8),
                                       ("bf16", torch.float32, 8), ("bf16", torch.float64, 16), ("f64", torch.float64, 8)])
def test_spmm_row_group_edges(n, val, dt, nb):
    import oracle as O
    from gen import ci_matrix, random_block
    from paper_2305_15552_gb300 import binding as B
    H = ci_matrix(n, 40, 64, seed=3, storage=val)
    X = torch.tensor(random_block(n, nb, seed=4), dtype=dt, device="cuda")
    P = B.SpmmPlan(H, layout="mirrored")
    Y = P.spmm(X).double().cpu().numpy()
    P.close()
    Xe = X.double().cpu().numpy()
    Ha = type(H)(n=n, rowptr=H.rowptr, col=H.col, val=np.abs(H.values_f64()), storage="f64")
    bound = O.sym_upper_matmul(Ha, np.abs(Xe))
    # rows of at most a few hundred terms: one rounding per multiply-add (FP32, FP64), 2^-44 per
    # double-float step
    eps = 2.0 ** -24 if dt == torch.float32 else (2.0 ** -53 if val == "f64" else 2.0 ** -44)
    assert np.all(np.abs(Y - O.sym_upper_matmul(H, Xe)) <= 300 * eps * bound + 1e-300)


# direct plans (FP64 values below 65,536 rows): fewer rows than a warp, a ragged last warp, one CTA
# round of the 152 SMs and a few CTAs more, the last size they take and the first they do not; every
# width, one column in place, the fused Chebyshev step, empty rows, rows without a diagonal
@pytest.mark.parametrize("n", [1, 33, 2500, 65535, 65536])
@pytest.mark.parametrize("nb", [1, 2, 4, 8, 16, 32])
def test_spmm_direct_edges(n, nb):
    import oracle as O
    from gen import ci_matrix, random_block
    from gen.synth import CSRUpper
    from paper_2305_15552_gb300 import binding as B
    H = ci_matrix(n, 30, 64, seed=5, storage="f64")
    rows = np.repeat(np.arange(n), np.diff(H.rowptr))
    keep = ~((rows % 7 == 3) & (H.col == rows)) & (rows % 11 != 5) & (H.col % 11 != 5)
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(rows[keep], minlength=n), out=rowptr[1:])
    H = CSRUpper(n=n, rowptr=rowptr, col=H.col[keep], val=H.val[keep], storage="f64")
    Xe = random_block(n, nb, seed=6)
    X = torch.tensor(Xe, device="cuda")
    P = B.SpmmPlan(H, layout="mirrored")
    Y = P.spmm(X).cpu().numpy()
    Ha = CSRUpper(n=n, rowptr=H.rowptr, col=H.col, val=np.abs(H.val), storage="f64")
    Yr, bound = O.sym_upper_matmul(H, Xe), O.sym_upper_matmul(Ha, np.abs(Xe))
    tol = 300 * 2.0 ** -53 * bound + 1e-300     # one rounding per multiply-add, rows of at most 300
    assert np.all(np.abs(Y - Yr) <= tol)
    if nb >= 8:
        Q = torch.tensor(random_block(n, nb, seed=7), device="cuda")
        act = torch.tensor([j % 3 != 1 for j in range(nb)], dtype=torch.int32, device="cuda")
        Z = P.spmm_cheb(X, 0.5, 2.0, Q, act).cpu().numpy()
        want = np.where(act.cpu().numpy() != 0, 0.5 * (Y - 2.0 * Xe) - Q.cpu().numpy(), Xe)
        # three roundings of the step on the same H X
        assert np.all(np.abs(Z - want) <= 4 * 2.0 ** -53 * (np.abs(Y) + 2 * np.abs(Xe) + np.abs(Q.cpu().numpy())))
    P.close()


# FP64 blocks on 16-byte but not on 32-byte boundaries: legal (rows move in pieces of at most 16 bytes), and
# the direct plans' gathers must then not take 32 bytes at once.  Each of X, Y and Qp is moved by itself
# and all together; the sums are those of the aligned call.
@pytest.mark.parametrize("n", [33, 2500])
@pytest.mark.parametrize("nb", [2, 4, 8, 16, 32])
def test_spmm_direct_16_byte_alignment(n, nb):
    import oracle as O
    from gen import ci_matrix, random_block
    from gen.synth import CSRUpper
    from paper_2305_15552_gb300 import binding as B

    def moved(a, by):
        v = torch.empty(a.size + by, dtype=torch.float64, device="cuda")[by:].view(a.shape)
        v.copy_(torch.tensor(a))
        assert v.data_ptr() % 32 == 8 * by
        return v

    H = ci_matrix(n, 30, 64, seed=5, storage="f64")
    Xe, Qe = random_block(n, nb, seed=6), random_block(n, nb, seed=7)
    Ha = CSRUpper(n=n, rowptr=H.rowptr, col=H.col, val=np.abs(H.val), storage="f64")
    Yr, bound = O.sym_upper_matmul(H, Xe), O.sym_upper_matmul(Ha, np.abs(Xe))
    P = B.SpmmPlan(H, layout="mirrored")
    Y0 = P.spmm(moved(Xe, 0))
    # one rounding per multiply-add, rows of at most 300
    assert np.all(np.abs(Y0.cpu().numpy() - Yr) <= 300 * 2.0 ** -53 * bound + 1e-300)
    act = torch.tensor([j % 3 != 1 for j in range(nb)], dtype=torch.int32, device="cuda")
    Z0 = P.spmm_cheb(moved(Xe, 0), 0.5, 2.0, moved(Qe, 0), act) if nb >= 8 else None
    for bx, by, bq in [(2, 0, 0), (0, 2, 0), (0, 0, 2), (2, 2, 2)]:
        assert torch.equal(P.spmm(moved(Xe, bx), moved(Xe, by)), Y0)
        if nb >= 8:
            assert torch.equal(P.spmm_cheb(moved(Xe, bx), 0.5, 2.0, moved(Qe, bq), act, Y=moved(Qe, by)), Z0)
    P.close()


# plan construction where it can go wrong: rows of more than 256 entries in a panel, row blocks of more
# than 32 upper tiles (two counting groups), a tile with few rows of many entries, columns whose entries
# all fall into one class mod 8, last row block and column block ragged
@pytest.mark.parametrize("val,dt", [("f32", torch.float32), ("bf16", torch.float32), ("f32", torch.float64)])
@pytest.mark.parametrize("kind", ["wide_rows", "one_class", "arrow"])
def test_plan_streams_edges(kind, val, dt):
    import oracle as O
    from gen import random_block
    from gen.synth import CSRUpper, round_to_storage
    from paper_2305_15552_gb300 import binding as B
    n = 9 * 256 + 37
    rng = np.random.default_rng(17)
    D = np.zeros((n, n), dtype=bool)
    np.fill_diagonal(D, rng.random(n) < 0.9)
    if kind == "wide_rows":
        D[5:20] |= rng.random((15, n)) < 0.7
        D[2000:2010] |= rng.random((10, n)) < 0.9
    elif kind == "one_class":
        D[:, 3::8] |= rng.random((n, D[:, 3::8].shape[1])) < 0.4
    else:
        D[:, -70:] = True
        D[0] = True
    D = np.triu(D)
    r, c = np.nonzero(D)
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(r, minlength=n), out=rowptr[1:])
    v = rng.standard_normal(r.size)
    H = CSRUpper(n=n, rowptr=rowptr, col=c.astype(np.int32), val=round_to_storage(v, val), storage=val)
    X = torch.tensor(random_block(n, 8, seed=9), dtype=dt, device="cuda")
    P = B.SpmmPlan(H, layout="mirrored")
    Y = P.spmm(X).double().cpu().numpy()
    P.close()
    Xe = X.double().cpu().numpy()
    Ha = CSRUpper(n=n, rowptr=rowptr, col=H.col, val=np.abs(H.values_f64()), storage="f64")
    bound = O.sym_upper_matmul(Ha, np.abs(Xe))
    # rows of at most n terms: one rounding of the running sum per term in FP32, 2^-44 in double-float
    eps = 2.0 ** -24 if dt == torch.float32 else 2.0 ** -44
    assert np.all(np.abs(Y - O.sym_upper_matmul(H, Xe)) <= n * eps * bound + 1e-300)


def _many_tiles(kind, n, rng):
    """Upper triangles whose row blocks have up to n / 64 tiles: row, column lists."""
    i = np.arange(n)
    r, c = [i], [i]
    if kind == "scattered":                 # a handful of entries per tile
        a, b = rng.integers(0, n, 30 * n), rng.integers(0, n, 30 * n)
        r += [np.minimum(a, b)]
        c += [np.maximum(a, b)]
    elif kind == "one_per_tile":            # the last column of every tile, the same for all rows
        for j in range(63, n, 64):
            k = i[i < j]
            r += [k]
            c += [np.full(k.size, j)]
    elif kind == "dense_rows":              # lengths around multiples of the 128 entries read at a time
        for x, m in [(3, n), (4, n), (300, 128), (301, 129), (302, 127), (303, 4096), (n - 400, 400)]:
            m = min(m, n - x)
            r += [np.full(m, x)]
            c += [np.arange(x, x + m)]
    else:                                   # "gaps": runs of 200 entries, 40 tiles without any between them
        for x in range(0, n, 37):
            k = np.concatenate([np.arange(q, min(q + 200, n)) for q in range(x, n, 64 * 40)])
            r += [np.full(k.size, x)]
            c += [k]
    key = np.unique(np.concatenate(r) * n + np.concatenate(c))
    return key // n, key % n


# row blocks of many tiles: several groups of 32 tiles in the column counts, rows left in the middle of a
# chunk of 128 entries and taken up again, panels by the dozen; small integers, so that every product is
# exact in any order
@pytest.mark.parametrize("kind", ["scattered", "one_per_tile", "dense_rows", "gaps"])
@pytest.mark.parametrize("val,dt", [("f32", torch.float32), ("bf16", torch.float32), ("f32", torch.float64),
                                    ("f64", torch.float64)])
@pytest.mark.parametrize("n", [9 * 256 + 37, 70000])
def test_plan_many_tiles_exact(kind, val, dt, n):
    import oracle as O
    from gen.synth import CSRUpper, round_to_storage
    from paper_2305_15552_gb300 import binding as B
    if kind == "one_per_tile" and n > 10000:
        n = 20480
    rng = np.random.default_rng(n)
    r, c = _many_tiles(kind, n, rng)
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(r, minlength=n), out=rowptr[1:])
    H = CSRUpper(n=n, rowptr=rowptr, col=c.astype(np.int32), val=round_to_storage(
        rng.integers(1, 4, r.size).astype(np.float64), val), storage=val)
    X = torch.tensor(rng.integers(-3, 4, (n, 8)), dtype=dt, device="cuda")
    P = B.SpmmPlan(H, layout="mirrored")
    Y = P.spmm(X).double().cpu().numpy()
    P.close()
    # sums of at most n products of magnitude 9: integers below 2^24
    assert 9 * n < 2 ** 24
    assert np.array_equal(Y, O.sym_upper_matmul(H, X.double().cpu().numpy()))


def test_plan_time_of_a_dense_row():
    """One dense row among 2M (31,250 tiles in one row block, 977 groups): the row is read once, not
    once per group.  Read once, the plan takes some tens of ms; once per group, 2 s and more."""
    import time
    from gen.synth import CSRUpper
    from paper_2305_15552_gb300 import binding as B
    n = 2_000_000
    rowptr = np.concatenate([[0], np.arange(n) + n]).astype(np.int64)
    col = np.concatenate([np.arange(n), np.arange(1, n)]).astype(np.int32)
    H = CSRUpper(n=n, rowptr=rowptr, col=col, val=np.ones(col.size, np.float32), storage="f32")
    dev = tuple(torch.tensor(a, device="cuda") for a in (H.rowptr, H.col, H.val))
    best = np.inf
    for _ in range(2):
        torch.cuda.synchronize()
        t = time.perf_counter()
        P = B.SpmmPlan(H, device_arrays=dev, layout="mirrored", copy=False)
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t)
        x = torch.ones(n, 1, device="cuda")
        y = P.spmm(x).cpu().numpy()[:, 0]
        P.close()
    want = np.full(n, 2.0)
    want[0] = n
    assert np.array_equal(y, want)
    assert best < 1.0, best


def test_plan_memory_of_scattered_entries():
    """1.2M tiles of 8 entries: the arrays over the tiles (0.6 GB) are gone before the streams (0.8 GB)
    are built, and no offset is kept per (tile, row) (1.3 GB).  With 1.9 GB left on the device the mirrored
    layout is built, and AUTO takes it."""
    import oracle as O
    from gen.synth import CSRUpper
    from paper_2305_15552_gb300 import binding as B
    n = 200_000
    rng = np.random.default_rng(2)
    a, b = rng.integers(0, n, 50 * n), rng.integers(0, n, 50 * n)
    key = np.unique(np.concatenate([np.minimum(a, b) * n + np.maximum(a, b), np.arange(n) * n + np.arange(n)]))
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(key // n, minlength=n), out=rowptr[1:])
    H = CSRUpper(n=n, rowptr=rowptr, col=(key % n).astype(np.int32), storage="f32",
                 val=rng.integers(1, 4, key.size).astype(np.float32))
    dev = tuple(torch.tensor(x, device="cuda") for x in (H.rowptr, H.col, H.val))
    X = torch.tensor(rng.integers(-3, 4, (n, 8)), dtype=torch.float32, device="cuda")
    Y = torch.empty_like(X)
    B.SpmmPlan(H, device_arrays=dev, layout="mirrored", copy=False).close()      # code loaded
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    rest = torch.empty(torch.cuda.mem_get_info()[0] - 1_900_000_000, dtype=torch.uint8, device="cuda")
    try:
        for layout in ("mirrored", "auto"):
            P = B.SpmmPlan(H, device_arrays=dev, layout=layout, copy=False)
            assert P.info()["layout"] == B.LAYOUTS["mirrored"]
            assert P.info()["n_tiles"] > 1_100_000
            P.spmm(X, Y)
            P.close()
            assert np.array_equal(Y.double().cpu().numpy(), O.sym_upper_matmul(H, X.double().cpu().numpy()))
    finally:
        del rest
        torch.cuda.empty_cache()


# more tiles than threads, so that a thread takes two (17, 34; 62 with itself) or four (31, 62) of them and
# one group takes the chunk: odd widths with 1 x 1 tiles, widths of 2 mod 4 with 2 x 2
@pytest.mark.parametrize("n", [31, 304 * 32 * 2 + 45])
@pytest.mark.parametrize("nb", [17, 31, 34, 62])
@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
def test_gram_several_tiles_a_thread(n, nb, dt):
    from paper_2305_15552_gb300 import binding as B
    rng = np.random.default_rng(n + nb)
    a, b = rng.standard_normal((n, nb)), rng.standard_normal((n, nb))
    A, Bm = torch.tensor(a, dtype=dt, device="cuda"), torch.tensor(b, dtype=dt, device="cuda")
    for X, Y in ((A, Bm), (A, A), (_shifted(a, dt), Bm)):
        G = B.gram(X, Y).cpu().numpy()
        Xe, Ye = X.double().cpu().numpy(), Y.double().cpu().numpy()
        # as in test_gram_chunk_edges
        tol = (2.0 ** -24 * 40 if dt == torch.float32 else 2.0 ** -53 * (n + 10)) * (np.abs(Xe).T @ np.abs(Ye)) + 1e-300
        assert np.all(np.abs(G - Xe.T @ Ye) <= tol)
        if X is Y:
            assert np.array_equal(G, G.T)


def test_plan_memory_of_half_layout():
    """16M rows: the tile bitmap (2.0 GB) is gone before the half-stored copy (0.6 GB) is built, so that
    2.4 GB are enough for the plan."""
    from gen.synth import CSRUpper
    from paper_2305_15552_gb300 import binding as B
    n = 16_000_000
    # the diagonal (2) and, for every row but the last 64, the column 64 to the right (1)
    rowptr = np.minimum(2 * np.arange(n + 1, dtype=np.int64), np.arange(n + 1, dtype=np.int64) + n - 64)
    i = np.arange(n, dtype=np.int64)
    col = np.empty(rowptr[-1], np.int32)
    val = np.full(rowptr[-1], 2.0)
    col[rowptr[:-1]] = i
    col[rowptr[:n - 64] + 1] = i[:n - 64] + 64
    val[rowptr[:n - 64] + 1] = 1.0
    H = CSRUpper(n=n, rowptr=rowptr, col=col, val=val, storage="f64")
    dev = tuple(torch.tensor(x, device="cuda") for x in (H.rowptr, H.col, H.val))
    x = torch.tensor(np.arange(n) % 7, dtype=torch.float64, device="cuda").reshape(n, 1)
    y = torch.empty_like(x)
    small = CSRUpper(n=64, rowptr=np.arange(65), col=np.arange(64, dtype=np.int32), val=np.ones(64), storage="f64")
    B.SpmmPlan(small, layout="half").close()      # code loaded
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    rest = torch.empty(torch.cuda.mem_get_info()[0] - 2_400_000_000, dtype=torch.uint8, device="cuda")
    try:
        P = B.SpmmPlan(H, device_arrays=dev, layout="half", copy=False)
    finally:
        del rest
        torch.cuda.empty_cache()
    assert P.info()["layout"] == B.LAYOUTS["half"]
    P.spmm(x, y)
    P.close()
    v = np.arange(n) % 7
    want = 2.0 * v
    want[:-64] += v[64:]
    want[64:] += v[:-64]
    assert np.array_equal(y.cpu().numpy()[:, 0], want)


# the lower triangle of full and nearly full tiles (an offset per tile and row; rows of more than the 24
# entries that the lanes keep in registers), either side of the mean fill from which it is built that way,
# with a ragged last row block and column block; small integers, exact in any order
@pytest.mark.parametrize("density", [0.15, 0.25, 0.6, 1.0])
@pytest.mark.parametrize("val,dt", [("f32", torch.float32), ("bf16", torch.float32), ("f64", torch.float64)])
@pytest.mark.parametrize("n", [300, 9 * 256 + 37])
def test_plan_dense_tiles_exact(density, val, dt, n):
    import oracle as O
    from gen.synth import CSRUpper, round_to_storage
    from paper_2305_15552_gb300 import binding as B
    rng = np.random.default_rng(n)
    D = np.triu(rng.random((n, n)) < density)
    D[np.arange(0, n, 5), np.arange(0, n, 5)] = False       # rows without a diagonal
    r, c = np.nonzero(D)
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(r, minlength=n), out=rowptr[1:])
    v = round_to_storage(rng.integers(1, 4, r.size).astype(np.float64), val)
    H = CSRUpper(n=n, rowptr=rowptr, col=c.astype(np.int32), val=v, storage=val)
    X = torch.tensor(rng.integers(-3, 4, (n, 8)), dtype=dt, device="cuda")
    P = B.SpmmPlan(H, layout="mirrored")
    Y = P.spmm(X).double().cpu().numpy()
    P.close()
    assert np.array_equal(Y, O.sym_upper_matmul(H, X.double().cpu().numpy()))
