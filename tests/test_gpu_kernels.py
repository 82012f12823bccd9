"""GPU kernels at the sizes where their splits can go wrong, against plain
FP64 arithmetic (numpy / torch)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1503_05464_gb300 as P
    return P


# one row; less than a tile; one past a panel and a tile, rows not 16-byte
# aligned; 96 columns (32-column chunks) at an odd offset; many chunks (more
# column chunks than the even split over the SMs handles in one wave); an
# uneven leaf that crosses tile boundaries
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("n,pad,c0,c1,starts", [
    (1, 0, 0, 1, None),
    (31, 5, 0, 3, [0, 31]),
    (129, 0, 0, 64, [0, 64, 129]),
    (193, 1, 0, 33, [0, 1, 100, 193]),
    (641, 3, 5, 101, [0, 320, 321, 641]),
    (400, 0, 0, 700, [0, 130, 390, 400]),
    (2100, 0, 0, 40, [0, 700, 1400, 2100]),
])
def test_simt_sampling_at_tile_edges(P, dtype, n, pad, c0, c1, starts):
    g = torch.Generator(device=DEV)
    g.manual_seed(n)
    A = torch.randn((n, n + pad), generator=g, device=DEV, dtype=torch.float64).to(dtype)[:, :n]
    R = torch.randn((n, c1), generator=g, device=DEV, dtype=torch.float64).to(dtype)
    Sr = torch.full((n, c1), 7.0, dtype=dtype, device=DEV)
    Sc = torch.full((n, c1), 7.0, dtype=dtype, device=DEV)
    P.hss_sample(A, R, c0, c1, Sr, Sc, leaf_starts=starts)
    only = torch.full((n, c1), 7.0, dtype=dtype, device=DEV)
    P.hss_sample(A, R, c0, c1, only, None, leaf_starts=starts)
    A64 = A.double().clone()
    for a, b in zip(starts or [], (starts or [])[1:]):
        A64[a:b, a:b] = 0.0
    X = R[:, c0:c1].double()
    # a length-n dot product: n roundings of |A||R|; 4 covers the compensation
    u = 2.0 ** -24 if dtype == torch.float32 else 2.0 ** -53
    for got, M in ((Sr, A64), (Sc, A64.T)):
        bound = 4 * n * u * (M.abs() @ X.abs())
        assert torch.all((got[:, c0:c1].double() - M @ X).abs() <= bound)
        assert torch.all(got[:, :c0] == 7.0)
    assert torch.equal(only, Sr)


# ranks on both sides of the 16-row tasks and of the 64-index stages, leaves
# at several depths, 1 to 33 columns (33: the level products)
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("n,leaf,rank,comb", [(300, 64, 7, False), (1030, 100, 17, False),
                                              (900, 150, 70, False), (500, 40, 16, True)])
def test_matvec_tasks_match_dense(P, dtype, n, leaf, rank, comb):
    import workloads as W
    A = torch.tensor(W.random_hss(n, leaf, rank, seed=n, diag_shift=20.0)[0], device=DEV).to(dtype)
    if comb:
        A = torch.tensor(W.toeplitz_inv_distance(n).numpy(), device=DEV).to(dtype)
    f64 = dtype == torch.float64
    tree = W.comb_tree_splits(n, leaf) if comb else None
    h = P.hss_compress(A, leaf_size=leaf, rtol=1e-11 if f64 else 1e-5, d0=rank + 20, d_step=32,
                       seed=3, tree=tree)
    g = torch.Generator(device=DEV).manual_seed(n)
    X = torch.randn(n, 33, dtype=torch.float64, device=DEV, generator=g).to(dtype)
    for k in (1, 3, 4, 9, 32, 33):
        Xs = torch.empty((n, k + 2), dtype=dtype, device=DEV)[:, :k].copy_(X[:, :k])   # ldx > nrhs
        Y = P.hss_matvec(h, Xs)
        ref = A.double() @ X[:, :k].double()
        err = float(torch.linalg.norm(Y.double() - ref) / torch.linalg.norm(ref))
        assert err <= (1e-9 if f64 else 1e-4), (k, err)
        assert torch.equal(P.hss_matvec(h, Xs), Y)


def test_matvec_of_nan_finishes(P):
    """An all-ones NaN (the work buffer's not-yet-written pattern) in x."""
    import time
    import workloads as W
    A = torch.as_tensor(W.toeplitz_inv_distance(1000), device=DEV)
    h = P.hss_compress(A, leaf_size=100)
    x = torch.ones(1000, dtype=torch.float64, device=DEV)
    x[::50] = torch.full((20,), -1, dtype=torch.int64, device=DEV).view(torch.float64)
    t = time.perf_counter()
    y = P.hss_matvec(h, x)
    torch.cuda.synchronize()
    assert time.perf_counter() - t < 1.0      # a poll gives up after about four seconds
    assert bool(torch.isnan(y).all())


# node orders on both sides of the per-node / blocked line (64 rows) and of
# the panels' cluster sizes (160, 320, 640 rows), partial last panels; the
# root's LU has to pivot (no diagonal shift)
@pytest.mark.parametrize("n,leaf,rank", [(260, 65, 31), (280, 70, 33), (640, 161, 75),
                                         (1300, 325, 130), (1400, 350, 321)])
def test_ulv_factor_solve_at_panel_edges(P, n, leaf, rank):
    import workloads as W
    A = W.random_hss(n, leaf, rank, seed=n)[0]
    h = P.hss_compress(torch.tensor(A, device=DEV), leaf_size=leaf, rtol=1e-13, d0=rank + 20,
                       d_step=32, seed=5)
    P.hss_factor(h)
    g = torch.Generator(device=DEV).manual_seed(n)
    b = torch.randn(n, 5, dtype=torch.float64, device=DEV, generator=g)
    x = P.hss_solve(h, b)
    # normwise backward error against the compressed form itself: 50 n u covers
    # the LQ and LU with a growth factor of order ten
    res = float(torch.linalg.norm(P.hss_matvec(h, x) - b))
    assert res <= 50 * n * 2.0 ** -53 * float(np.linalg.norm(A)) * float(torch.linalg.norm(x))
    P.hss_factor(h)
    assert torch.equal(P.hss_solve(h, b), x)


# few to many row blocks per launch: the update takes blocks of 8, 16, 24 or 32
# rows, and a row's sums must not depend on it
def test_ulv_factors_whatever_shares_the_launch(P):
    import workloads as W
    A = W.random_hss(1400, 350, 300, seed=9)[0]
    At = torch.tensor(A, device=DEV)
    hs = [P.hss_compress(At, leaf_size=350, rtol=1e-13, d0=320, d_step=32, seed=5) for _ in range(17)]
    b = torch.randn(1400, 3, dtype=torch.float64, device=DEV,
                    generator=torch.Generator(device=DEV).manual_seed(1))
    P.hss_factor(hs[0])
    x = P.hss_solve(hs[0], b)
    for count in (2, 3, 5, 17):
        P.hss_factor_batched(hs[:count])
        for h in hs[:count]:
            assert torch.equal(P.hss_solve(h, b), x)


# one column to more than a launch's 64 (two slabs), in place, on handles with
# 8-row tasks (nodes above 160 rows), partial blocks, rank-zero nodes and a
# single-node tree; several handles of different widths together
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_ulv_solve_tasks(P, dtype):
    import scipy.linalg as sla
    import workloads as W
    mats = [(W.random_hss(900, 225, 90, seed=1, diag_shift=60.0)[0], 225, 110),
            (W.random_hss(130, 64, 33, seed=2, diag_shift=30.0)[0], 64, 45),
            (sla.block_diag(*[np.eye(40) * (i + 2) for i in range(5)]), 40, 16),
            (np.random.default_rng(3).standard_normal((70, 70)) + 20 * np.eye(70), 128, 16)]
    f64 = dtype == torch.float64
    hs, norms = [], []
    for A, leaf, d0 in mats:
        At = torch.tensor(A, device=DEV).to(dtype)
        norms.append(float(np.linalg.norm(A)))
        hs.append(P.hss_compress(At, leaf_size=leaf, rtol=1e-12 if f64 else 1e-6, d0=d0, d_step=16, seed=4))
        P.hss_factor(hs[-1])
    g = torch.Generator(device=DEV).manual_seed(9)
    Bs = []
    for h, nA, k in zip(hs, norms, (70, 3, 1, 9)):
        B = torch.randn(h.n, k, dtype=torch.float64, device=DEV, generator=g).to(dtype)
        X = P.hss_solve(h, B)
        # normwise backward error against the compressed form: FP64 as in the
        # test above; FP32 the product's own bound (length-n FP32 sums)
        bound = (50 * 2.0 ** -53 if f64 else 4 * 2.0 ** -24) * h.n * nA * float(torch.linalg.norm(X.double()))
        Y = torch.cat([P.hss_matvec(h, X[:, c:c + 32].contiguous()) for c in range(0, k, 32)], 1)
        assert float(torch.linalg.norm(Y.double() - B.double())) <= bound
        for c in {0, k - 1}:         # a column's bits do not depend on the others
            assert torch.equal(P.hss_solve(h, B[:, c].contiguous()), X[:, c])
        Y = B.clone()
        assert torch.equal(P.hss_solve(h, Y, X=Y), X)
        Bs.append(B)
    Xs, st = P.hss_solve_batched(hs, Bs)
    assert st == [0] * 4
    for h, B, X in zip(hs, Bs, Xs):
        assert torch.equal(P.hss_solve(h, B), X)


# one column; k at, below and above a block of 16 rows of the back
# substitution; fewer, as many and more columns than a warp; short columns
# (the shared blocks larger than a column) and long ones; columns in shared
# and (the last) in global memory; k = min(m, d), nothing left for E
@pytest.mark.parametrize("d,m,k", [
    (17, 1, 1), (16, 33, 16), (40, 31, 15), (40, 33, 17), (127, 65, 31), (129, 200, 33),
    (401, 90, 48), (64, 520, 60), (33, 20, 20), (900, 700, 97),
])
def test_id_at_block_edges(P, d, m, k):
    """Against the oracle's CPQR: the same pivots (random matrices of exact
    rank: residual norms differ far above rounding) and generators (the
    triangle's condition is below 1e5, so its rounding below 1e-10)."""
    from oracle import hss_oracle as O
    rng = np.random.default_rng(1000 * d + m)
    Y = rng.standard_normal((d, k)) @ rng.standard_normal((k, m))
    r = O.interpolative_decomposition(Y, 1e-11)
    Yt = torch.tensor(Y.T.copy(), dtype=torch.float64, device=DEV)
    for copies in (1, 7):   # alone, and in a batch (other clusters, the same bits)
        for kg, perm, E in P.hss_id_batched([Yt] * copies, 1e-11):
            perm = perm.cpu().numpy()
            assert kg == r.k == k
            assert list(perm[:k]) == list(r.perm[:k])
            assert sorted(perm.tolist()) == list(range(m))
            G = np.zeros((m, k))
            G[perm[:k]] = np.eye(k)
            G[perm[k:]] = E.cpu().numpy().reshape(m - k, k)
            np.testing.assert_allclose(G, r.basis(), rtol=1e-7, atol=1e-9)


@pytest.mark.parametrize("d,m", [(40, 30), (300, 500)])
def test_id_of_nan_finishes(P, d, m):
    Y = torch.full((m, d), float("nan"), dtype=torch.float64, device=DEV)
    k, perm, _ = P.hss_id_batched([Y], 1e-6)[0]
    assert 0 <= k <= min(m, d)
    assert sorted(perm.cpu().tolist()) == list(range(m))


# one tile; a pair's phantom second panel; clusters whose range crosses panel
# pairs (R_p changes, the exchange through its buffer drains first), ragged
# tiles, one column, a second 64-column box, the full width, two sweeps
@pytest.mark.parametrize("mode,tol", [("bf16x3", 1e-5), ("bf16x2", 3e-5), ("tf32", 5.2e-4)])
@pytest.mark.parametrize("n,c,starts", [
    (60, 7, None), (129, 1, [0, 100, 129]), (700, 65, None), (2000, 128, [0, 700, 701, 2000]),
    (2003, 131, None), (3500, 33, [0, 1000, 3500]),
])
def test_tensor_core_sampling_at_segment_edges(P, mode, tol, n, c, starts):
    """Against FP64, and the same bits on every repeat.  Bound, relative to
    |A| |R|: the split's 2^-24 / 2^-16 / 2^-11 and at most 80 FP32 roundings
    (2^-23 each: the tensor core truncates)."""
    pitch = (n + 3) // 4 * 4
    rng = np.random.default_rng(n + c)
    A = torch.tensor(rng.standard_normal((n, pitch)), dtype=torch.float32, device=DEV)[:, :n]
    R = torch.zeros((n, c), device=DEV)
    P.hss_random_gaussian(3, n, 0, c, R)
    A64, R64 = A.double(), R.double()
    if starts is not None:
        A64 = A64.clone()
        for lo, hi in zip(starts[:-1], starts[1:]):
            A64[lo:hi, lo:hi] = 0
    first = None
    for _ in range(6):
        Sr = torch.empty((n, c), device=DEV)
        Sc = torch.empty((n, c), device=DEV)
        P.hss_sample(A, R, 0, c, Sr, Sc, leaf_starts=starts, mode=mode)
        if first is None:
            first = (Sr, Sc)
        assert torch.equal(Sr, first[0]) and torch.equal(Sc, first[1])
    for M, S in ((A64, Sr), (A64.T, Sc)):
        bound = tol * (M.abs() @ R64.abs()) + 1e-30
        assert bool(((S.double() - M @ R64).abs() <= bound).all())


# products of one tile and of many (tiles of 16, 32 and 64 rows), ragged rows,
# columns and inner lengths: a factorization's D, Vhat, W and root updates
@pytest.mark.parametrize("n,leaf,rank", [(131, 66, 5), (530, 133, 49), (2100, 525, 130), (3300, 413, 71)])
def test_ulv_products_at_tile_edges(P, n, leaf, rank):
    import workloads as W
    A = W.random_hss(n, leaf, rank, seed=n, diag_shift=float(n))[0]
    h = P.hss_compress(torch.tensor(A, device=DEV), leaf_size=leaf, rtol=1e-13, d0=rank + 20,
                       d_step=32, seed=5)
    P.hss_factor(h)
    b = torch.randn(n, 2, dtype=torch.float64, device=DEV,
                    generator=torch.Generator(device=DEV).manual_seed(n))
    x = P.hss_solve(h, b)
    # normwise backward error against the compressed form itself: 50 n u covers
    # the LQ and LU with a growth factor of order ten
    res = float(torch.linalg.norm(P.hss_matvec(h, x) - b))
    assert res <= 50 * n * 2.0 ** -53 * float(np.linalg.norm(A)) * float(torch.linalg.norm(x))


# sweeps of one call that differ in width (65 + 66 columns, 86 + 87 + 87, 106 +
# 107 + 107) share the leaf mask; the last is as wide as a 128-column sweep gets
@pytest.mark.parametrize("mode,tol", [("bf16x3", 1e-5), ("bf16x2", 3e-5), ("tf32", 5.2e-4)])
@pytest.mark.parametrize("c", [131, 260, 320, 383])
def test_tensor_core_sampling_masks_every_sweep(P, mode, tol, c):
    n, starts = 1100, [0, 300, 301, 700, 1100]
    rng = np.random.default_rng(c)
    A = torch.tensor(rng.standard_normal((n, n)), dtype=torch.float32, device=DEV)
    R = torch.zeros((n, c), device=DEV)
    P.hss_random_gaussian(3, n, 0, c, R)
    M = A.double()
    for lo, hi in zip(starts[:-1], starts[1:]):
        M[lo:hi, lo:hi] = 0
    Sr, Sc, only = (torch.empty((n, c), device=DEV) for _ in range(3))
    P.hss_sample(A, R, 0, c, Sr, Sc, leaf_starts=starts, mode=mode)
    P.hss_sample(A, R, 0, c, only, None, leaf_starts=starts, mode=mode)
    assert torch.equal(only, Sr)
    R64 = R.double()
    for W, S in ((M, Sr), (M.T, Sc)):   # the bound of the test above
        assert bool(((S.double() - W @ R64).abs() <= tol * (W.abs() @ R64.abs()) + 1e-30).all())


# a NaN leaves no pivot in some column of the root's LU: in one CTA (50 rows),
# blocked over 1 to 8 CTAs, and from a leaf block below the root
@pytest.mark.parametrize("n,leaf", [(50, 64), (63, 64), (64, 64), (100, 128), (300, 512), (700, 1024),
                                    (100, 50), (400, 100)])
@pytest.mark.parametrize("at", [(0, 0), (-1, -1), (3, 20)])
def test_factor_of_nan_is_singular(P, n, leaf, at):
    import workloads as W
    A = torch.as_tensor(W.toeplitz_inv_distance(n), device=DEV).clone()
    good = P.hss_compress(A, leaf_size=leaf)
    A[at] = float("nan")          # (the sampling masks the leaf blocks: ranks as without it)
    h = P.hss_compress(A, leaf_size=leaf)
    with pytest.raises(P.HssError) as e:
        P.hss_factor(h)
    assert e.value.status == P.hss.HSS_ERR_SINGULAR
    with pytest.raises(P.HssError) as e:
        P.hss_solve(h, torch.ones(n, dtype=torch.float64, device=DEV))
    assert e.value.status == P.hss.HSS_ERR_STATE
    assert P.hss_factor_batched([h, good]) == [P.hss.HSS_ERR_SINGULAR, 0]
    # the other handle's solution: |A - H| <= 100 rtol |A|, condition below 3
    b = torch.ones(n, dtype=torch.float64, device=DEV)
    A = torch.as_tensor(W.toeplitz_inv_distance(n), device=DEV)
    assert float((A @ P.hss_solve(good, b) - b).norm()) <= 3e-4 * float(b.norm())


def test_id_launch_choice_fits_every_shape_of_a_class(P):
    """Two batches of one tuner class (powers of two of their sizes), in
    clusters of 8, which may double, and of 16, which may not; both through
    the whole of the class's trials."""
    def batch(count, m, d, seed):
        g = torch.Generator(device=DEV).manual_seed(seed)
        B = torch.randn(20, d, generator=g, device=DEV, dtype=torch.float64)
        return [torch.randn(m, 20, generator=g, device=DEV, dtype=torch.float64) @ B for _ in range(count)]
    pair = batch(10, 517, 384, 1), batch(8, 755, 496, 2)
    first = [P.hss_id_batched(Y, 1e-9) for Y in pair]
    for _ in range(8):
        for Y, ref in zip(pair, first):
            for x, y in zip(P.hss_id_batched(Y, 1e-9), ref):
                assert x[0] == y[0] == 20 and torch.equal(x[1], y[1]) and torch.equal(x[2], y[2])


# panel partials (128 rows each) whose running sum leaves FP32's range and comes
# back: 3e38 + 3e38 - 3e38 - 2e38; an odd pitch with bf16x3 takes the mma.sync
# kernel
@pytest.mark.parametrize("mode,pad", [("native", 0), ("native", 1), ("bf16x3", 1)])
def test_column_sample_whose_partials_pass_the_fp32_range(P, mode, pad):
    n, c = 600, 5
    A = torch.zeros((n, n + pad), device=DEV)[:, :n]
    for i, v in ((3, 3e38), (130, 3e38), (257, -3e38), (400, -2e38)):
        A[i] = v
    A[:, 7] = 0.0
    A[500, 7] = float("inf")
    A[501, 8] = float("nan")
    R = torch.ones((n, c), device=DEV)
    Sr, Sc = torch.empty((n, c), device=DEV), torch.empty((n, c), device=DEV)
    P.hss_sample(A, R, 0, c, Sr, Sc, mode=mode)
    want = A.double().T @ R.double()
    plain = [j for j in range(n) if j not in (7, 8)]
    # one rounding of each term (bf16x3: its three planes hold 24 bits) and of the sum
    assert bool(((Sc.double() - want)[plain].abs() <= 5 * 2.0 ** -23 * 3e38).all())
    assert bool(torch.isnan(Sc[8]).all())
    if mode == "native":
        assert bool((Sc[7] == float("inf")).all())


def test_row_sample_keeps_the_remainders_at_cuts(P):
    """FP32, rows of A against ones: 2^23, then 124 times 0.75 (one in each
    tile), so that every sum rounds and the remainders carry the rest.  The
    CTAs' ranges cut a row's panel two or three times, each panel elsewhere;
    the total, 2^23 + 93, is a number of FP32."""
    n = 8000          # 63 panels of 125 tiles on 152 SMs
    A = torch.zeros((n, n), device=DEV)
    A[:, ::64] = 0.75
    A[:, 0] = 2.0 ** 23
    R = torch.ones((n, 3), device=DEV)
    S = torch.empty((n, 3), device=DEV)
    P.hss_sample(A, R, 0, 3, S, None)
    assert bool((S == 2.0 ** 23 + 93).all())


# the most columns 16 CTAs hold beside few samples (their shared memory is full);
# many columns and few samples, so that the back substitution's block takes the
# columns' own arrays; and beside smaller items, whose block has doubles of its own
@pytest.mark.parametrize("shapes", [[(76400, 32)], [(75700, 128)], [(3000, 40)], [(2200, 399), (60, 33), (130, 140)]])
def test_id_of_many_columns_and_few_samples(P, shapes):
    g = torch.Generator(device=DEV).manual_seed(len(shapes))
    k, Ys = 19, []
    for m, d in shapes:
        B = torch.randn(k, d, generator=g, device=DEV, dtype=torch.float64)
        Ys.append(torch.randn(m, k, generator=g, device=DEV, dtype=torch.float64) @ B)
    out = P.hss_id_batched(Ys, 1e-9)
    for Y, (kk, perm, E) in zip(Ys, out):
        m = Y.shape[0]
        assert kk == k
        assert torch.equal(torch.sort(perm).values, torch.arange(m, device=DEV, dtype=torch.int32))
        perm = perm.long()
        # Y's other rows from the skeleton rows: E's entries are a few units, k
        # roundings of each product, and the triangle's condition below 1e5
        assert float((Y[perm[k:]] - E @ Y[perm[:k]]).abs().max()) <= 1e-9 * float(Y.abs().max())
        kk1, perm1, E1 = P.hss_id_batched([Y], 1e-9)[0]
        assert kk1 == k and torch.equal(perm1.long(), perm) and torch.equal(E1, E)


def _ill_triangles(kind, n, seed):
    """A = L U with |B||B^-1| to 1e11 in its diagonal blocks, and |L||U|: unit
    lower triangles of -0.9 (partial pivoting keeps the rows), or U alone, or U
    with two diagonal entries 2^120 below their rows."""
    rng = np.random.default_rng(seed)
    low = np.tril(-0.9 * np.ones((n, n)), -1) + np.eye(n)
    up = np.triu(rng.standard_normal((n, n)), 1) + 6 * np.eye(n)
    if kind != "lower":
        low, up = np.eye(n), np.triu(-np.ones((n, n)), 1) + np.eye(n)
    if kind == "wide":
        up[3, 3] = up[n - 2, n - 2] = 2.0 ** -120
    return low @ up, np.abs(low) @ np.abs(up)


def _solves_as_substitution(P, A, bound, leaf):
    """|A x - b| within `bound` |x| and a column's bits the same in every
    width (1, 2 and 4 columns a task) and in a batch."""
    n = A.shape[0]
    h = P.hss_compress(torch.tensor(A, device=DEV), leaf_size=leaf)
    P.hss_factor(h)
    b = A @ np.random.default_rng(n).standard_normal((n, 33))
    B = torch.tensor(b, device=DEV)
    x = P.hss_solve(h, B)
    xn = x.cpu().numpy()
    assert np.all(np.abs(A @ xn - b) <= bound(xn))
    for k in (1, 9):
        assert torch.equal(P.hss_solve(h, B[:, :k].contiguous()), x[:, :k])
    X, st = P.hss_solve_batched([h, h], [B[:, :3].contiguous(), B])
    assert st == [0, 0] and torch.equal(X[0], x[:, :3]) and torch.equal(X[1], x)


@pytest.mark.parametrize("kind", ["lower", "upper", "wide"])
@pytest.mark.parametrize("n", [20, 33, 45, 60])
def test_solve_with_ill_conditioned_root_blocks(P, kind, n):
    A, LU = _ill_triangles(kind, n, n)
    # Higham, Accuracy and Stability, theorem 9.4: 3 n u |L||U||x|
    _solves_as_substitution(P, A, lambda x: 3 * n * 2.0 ** -53 * (LU @ np.abs(x)), 128)


@pytest.mark.parametrize("n", [20, 45, 64, 150])
def test_solve_with_ill_conditioned_node_blocks(P, n):
    """Two nodes of rank zero, each A_i = L Q: the LQ's L is ill conditioned.
    Householder LQ and substitution: 10 n u |A||x| in norms."""
    import scipy.linalg as sla
    rng = np.random.default_rng(n)
    low = np.tril(-0.9 * np.ones((n, n)), -1) + np.eye(n)
    A = sla.block_diag(*[low @ np.linalg.qr(rng.standard_normal((n, n)))[0] for _ in range(2)])
    _solves_as_substitution(
        P, A, lambda x: 10 * n * 2.0 ** -53 * np.linalg.norm(A) * np.linalg.norm(x, axis=0), n)


@pytest.mark.parametrize("kind", ["lower", "upper"])
@pytest.mark.parametrize("n", [64, 100, 150, 333])
def test_factor_with_ill_conditioned_panels(P, kind, n):
    """The same triangles down the diagonal of a blocked root: the panels' unit
    triangles are ill conditioned too."""
    import scipy.linalg as sla
    As, LUs = zip(*[_ill_triangles(kind, min(60, n - i), i) for i in range(0, n, 60)])
    A, LU = sla.block_diag(*As), sla.block_diag(*LUs)
    _solves_as_substitution(P, A, lambda x: 3 * n * 2.0 ** -53 * (LU @ np.abs(x)), 512)


# a single node: fewer CTAs per SM than fit, one and several rounds of tasks
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("n", [90, 1000, 2600, 5200])
def test_matvec_of_one_dense_node(P, dtype, n):
    g = torch.Generator(device=DEV).manual_seed(n)
    A = torch.randn(n, n, generator=g, device=DEV, dtype=torch.float64).to(dtype)
    X = torch.randn(n, 32, generator=g, device=DEV, dtype=torch.float64).to(dtype)
    h = P.hss_compress(A, leaf_size=n)
    full = P.hss_matvec(h, X)
    # a sum of n products
    u = 2.0 ** -24 if dtype == torch.float32 else 2.0 ** -53
    A64, X64 = A.double(), X.double()
    assert bool(((full.double() - A64 @ X64).abs() <= 2 * n * u * (A64.abs() @ X64.abs())).all())
    for k in (1, 3, 9):
        x = X[:, :k].contiguous()
        y = P.hss_matvec(h, x)
        assert torch.equal(y, full[:, :k]) and torch.equal(P.hss_matvec(h, x), y)


# the root's interchanges fit shared memory up to 2112 rows
@pytest.mark.parametrize("n", [2112, 2113])
def test_root_interchanges_on_both_sides_of_shared_memory(P, n):
    g = torch.Generator(device=DEV).manual_seed(n)
    A = torch.randn(n, n, generator=g, device=DEV, dtype=torch.float64)
    h = P.hss_compress(A, leaf_size=n)
    P.hss_factor(h)
    b = torch.randn(n, 2, generator=g, device=DEV, dtype=torch.float64)
    x = P.hss_solve(h, b)
    # partial pivoting: growth below 50 on random matrices, n u each
    assert float((A @ x - b).norm()) <= 50 * n * 2.0 ** -53 * float(A.norm()) * float(x.norm())
