"""The block-row kernels with triples of lanes (codes 401, 402, 404, 408) and
the CTAs of long rows: against the block product's definition and the oracle's
V-cycle."""
import numpy as np
import pytest

import fsi_inputs as F
from oracle import amg
from oracle.sparse import to_csr

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2206_06996_gb300 as pkg  # noqa: E402

pkg.load_library(build_if_missing=True)

CODES = (401, 402, 404, 408)


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _random(rng, nbr, nbc, longest):
    k = rng.integers(0, longest + 1, nbr)
    k[nbr // 2] = min(longest, nbc)
    rows = [np.sort(rng.choice(nbc, size=min(n, nbc), replace=False)) for n in k]
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    return F.BSR(3, 3, nbr, nbc, rp, np.concatenate(rows).astype(np.int32), rng.standard_normal(int(rp[-1]) * 9))


@pytest.mark.parametrize("code", CODES)
@pytest.mark.parametrize("nbr", [1, 9, 10, 79, 80, 81, 1217])
def test_triples_of_lanes_equal_the_product(code, nbr):
    """Sizes around a warp's rows (1, 2, 5, 10) and a CTA's (8 to 80), rows of
    0 to 31 blocks (odd remainders of 3 to 30 lanes).  A row sums at most 93
    products: each is off by eps/2 and each partial sum by eps/2 of at most the
    absolute sum, so the error is below 94 * 1.2e-16 * sum |a x|."""
    rng = np.random.default_rng(nbr + code)
    M = _random(rng, nbr, max(nbr, 31), 31)
    x = rng.standard_normal(M.nb_cols * 3)
    with pkg.BlockSolver(spmv_group=code, autotune=0):
        y = pkg.bsr_spmv(pkg.DeviceBSR.from_host(M), _dev(x)).cpu().numpy()
    A = to_csr(M)
    bound = 94 * 1.2e-16 * (abs(A) @ np.abs(x))
    assert np.all(np.abs(y - A @ x) <= bound + 1e-300)


@pytest.mark.parametrize("code", CODES + (102, 302, 304))
def test_vcycle_with_long_rows_matches_oracle(code):
    """On the small tube the axis nodes' rows (75 blocks among rows of 15) are
    summed by CTAs of their own: V-cycles of A with every epilogue equal the
    oracle's on the exported hierarchy."""
    s = F.tube_system("tube_small")
    assert np.diff(s.A.row_ptr).max() > 3 * s.A.nnzb // s.n_v
    with pkg.BlockSolver(spmv_group=code, autotune=0) as sol:
        sol.setup(s.A, s.B, s.C, s.D)
        nl = sol.amg_levels(pkg.SCR_HIER_A)
        As = [to_csr(sol.export(pkg.SCR_HIER_A, l, pkg.SCR_EXPORT_OPERATOR)) for l in range(nl)]
        Ps = [to_csr(sol.export(pkg.SCR_HIER_A, l, pkg.SCR_EXPORT_PROLONGATOR)) for l in range(nl - 1)]
        b = np.random.default_rng(code).standard_normal(As[0].shape[0])
        x = sol.amg_apply(pkg.SCR_HIER_A, _dev(b)).cpu().numpy()
    ref = amg.vcycle(amg.hierarchy_from_matrices(As, Ps, 3, 1, 1, "cheb", 3), b)
    assert np.linalg.norm(x - ref) <= 1e-11 * np.linalg.norm(ref)


@pytest.mark.parametrize("preset,which,bs", [("tube_tiny", pkg.SCR_HIER_A, 3), ("tube_mini", pkg.SCR_HIER_SHAT, 1),
                                             ("tube_mini", pkg.SCR_HIER_A, 3)])
def test_dense_coarsest_solve_inverts_the_operator(preset, which, bs):
    """A hierarchy of one level is the dense inverse alone: 81 and 949 rows in
    one cluster's shared memory or in L2, 2,379 rows in L2; x = A^{-1} b has
    the residual of an explicit inverse, at most 8 n eps cond(A) |b|."""
    s = F.tube_system(preset)
    with pkg.BlockSolver(amg_max_levels=1) as sol:
        sol.setup(s.A, s.B, s.C, s.D)
        A = to_csr(sol.export(which, 0, pkg.SCR_EXPORT_OPERATOR)).toarray()
        n = A.shape[0]
        b = np.random.default_rng(n).standard_normal(n)
        x = sol.amg_apply(which, _dev(b)).cpu().numpy()
    tol = 8 * n * np.finfo(float).eps * np.linalg.cond(A)
    assert np.linalg.norm(A @ x - b) <= tol * np.linalg.norm(b)


@pytest.mark.parametrize("precision", [pkg.SCR_FP64, pkg.SCR_MIXED])
@pytest.mark.parametrize("sets", [1, 2, 4, 8])
def test_eight_column_products_solve_every_column(precision, sets):
    """The eight-column kernels with 1, 2, 4 and 8 lane sets per block row
    (every block shape and epilogue of the block solve, long rows among them):
    each column's residual, recomputed by the oracle, meets the solve's
    tolerance."""
    s = F.tube_system("tube_mini")
    rng = np.random.default_rng(sets)
    xs = [rng.standard_normal(s.n) * (c + 1) for c in range(8)]
    from oracle.sparse import BlockOperator
    op = BlockOperator.from_system(s)
    bs = [op.matvec(x) for x in xs]
    with pkg.BlockSolver(nrhs=8, precision=precision, spmv_group=100 + sets, autotune=0) as sol:
        sol.setup(s.A, s.B, s.C, s.D)
        got, rel = sol.solve_multi([_dev(b) for b in bs])
    for c in range(8):
        x = got[c].cpu().numpy()
        assert rel[c] <= 1e-8 and np.linalg.norm(op.matvec(x) - bs[c]) <= 1.001e-8 * np.linalg.norm(bs[c])


# ------------------------------------------------- eight columns and one column
def _listed(M):
    """Block rows that get a CTA of their own: more than max(32, 3 x the mean)
    blocks, where these are at most max(64, rows / 512)."""
    k = np.diff(M.row_ptr)
    n = int((k > max(32, 3 * (len(M.col) // M.nb_rows))).sum())
    return n if n <= max(64, M.nb_rows // 512) else 0


@pytest.mark.parametrize("precision,tol", [(pkg.SCR_FP64, 1e-10), (pkg.SCR_MIXED, 1e-3)])
@pytest.mark.parametrize("sets", [1, 2, 4, 8])
def test_eight_columns_take_the_steps_of_one(precision, tol, sets):
    """Eight multiples 2^c b of one right-hand side span the Krylov spaces of b
    alone: with every inner solve cut after a fixed number of steps and one outer
    step, column c of the block solve is 2^c times the one-column solve's result,
    which every product, restriction, prolongation and smoothing step of both
    hierarchies enters.  A, B, C and D list long rows here.  About 200 products
    in a chain, each off by a few eps and those errors grown by a factor of 100
    at most: 1e-10 in FP64; 1e-3 with FP32 sums (and BF16 coarse values, the same
    on both sides)."""
    s = F.tube_system("tube_small")
    assert all(_listed(M) for M in (s.A, s.B, s.C, s.D))
    opts = dict(precision=precision, autotune=0, max_it=1, max_A=3, max_S=2, max_I=2, rtol_A=1e-30, rtol_S=1e-30,
                rtol_I=1e-30)
    shift = [3, -2, 0, 4, 1, -1, 2, -3]
    with pkg.BlockSolver(spmv_group=102, **opts) as sol:
        sol.setup(s.A, s.B, s.C, s.D)
        assert _listed(sol.export(pkg.SCR_HIER_A, 1, pkg.SCR_EXPORT_OPERATOR))  # BF16 values in mixed precision
        x = sol.solve(s.b.copy(), raise_on_nonconvergence=False)
        one = {k: v for k, v in sol.stats().items() if k in ("a_iters", "s_iters", "i_iters", "outer_iters")}
    with pkg.BlockSolver(nrhs=8, spmv_group=100 + sets, **opts) as sol:
        sol.setup(s.A, s.B, s.C, s.D)
        got, _ = sol.solve_multi([s.b * 2.0 ** c for c in shift], raise_on_nonconvergence=False)
        assert {k: v for k, v in sol.stats().items() if k in one} == one
    for c, y in zip(shift, got):
        assert np.linalg.norm(y * 2.0 ** -c - x) <= tol * np.linalg.norm(x)


# ------------------------------------------------------------- crafted systems
def _bsr(br, bc, rows, nbc, value):
    """Block matrix of per-row column lists, value(row, column) -> br x bc."""
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    col = np.array([c for r in rows for c in r], np.int32)
    val = [np.asarray(value(i, c), float).reshape(-1) for i, r in enumerate(rows) for c in r]
    return F.BSR(br, bc, len(rows), nbc, rp, col, np.concatenate(val) if val else np.zeros(0))


def _identity(br, n, scale=1.0):
    return _bsr(br, br, [[i] for i in range(n)], n, lambda i, c: scale * np.eye(br))


def _none(br, bc, nbr, nbc):
    """A matrix of one stored zero block."""
    return _bsr(br, bc, [[0]] + [[]] * (nbr - 1), nbc, lambda i, c: np.zeros((br, bc)))


def test_sparse_product_rows_around_its_table_sizes():
    """Shat = D - C B for A = I and whole numbers is exact, and so is its numeric
    refresh: rows of C B with 1 to 700 columns, 511, 512, 513 (the numeric pass
    with sums in shared memory ends at 512) and upper bounds of 504, 512, 513 and
    more (the symbolic pass takes a table in global memory above 512) among them,
    from rows of C with up to 200 blocks (chunks of 32)."""
    rng = np.random.default_rng(5)
    q, n = 140, 703  # B: q rows of eight columns (three of them shared with the next), then one column each
    brow = [list(range(5 * j, 5 * j + 8)) for j in range(q)] + [[i] for i in range(n)]
    want = [1, 3, 8, 31, 32, 33, 63, 64, 65, 318, 323, 324, 325, 508, 510, 511, 512, 513, 514, 600, 700]
    crow = []
    for i in range(n):
        m = want[i % len(want)] if i < 3 * len(want) else int(rng.integers(0, 40))
        chunks = max(0, (m - 3) // 5) if i % 2 == 0 else 0
        first = 5 * chunks + 3 if chunks else 0
        singles = range(first, m if m <= 200 or chunks else 200)
        crow.append(list(range(chunks)) + [q + c for c in singles])
    lengths = [len(set(c for v in r for c in brow[v])) for r in crow]
    bounds = [sum(len(brow[v]) for v in r) for r in crow]
    assert {511, 512, 513} <= set(lengths) and {504, 512} <= set(bounds) and max(map(len, crow)) > 128
    whole = lambda r, c: (lambda i, j: rng.integers(-8, 9, (r, c)) * 1.0)
    B, C = _bsr(3, 1, brow, n, whole(3, 1)), _bsr(1, 3, crow, q + n, whole(1, 3))
    D = _identity(1, n, 2.0 ** 20)
    A = _identity(3, q + n)
    with pkg.BlockSolver(autotune=0) as sol:
        sol.setup(A, B, C, D)
        for again in range(2):
            if again:
                B, C = (F.BSR(M.br, M.bc, M.nb_rows, M.nb_cols, M.row_ptr, M.col,
                              rng.integers(-8, 9, M.val.size) * 1.0) for M in (B, C))
                sol.update_values(A, B, C, D)
            S = to_csr(sol.export(pkg.SCR_HIER_SHAT, 0, pkg.SCR_EXPORT_OPERATOR))
            assert np.array_equal(S.toarray(), (to_csr(D) - to_csr(C) @ to_csr(B)).toarray())


def test_block_sparse_products_with_wide_rows():
    """3x3 products whose rows have fewer and more than 64 blocks (sums in shared
    memory up to there) from rows of 3 to 420 blocks: prolongators and Galerkin
    operators equal the oracle's of the exported aggregates."""
    n, rng = 420, np.random.default_rng(6)
    rows = [sorted({(i - 1) % n, i, (i + 1) % n} | set(range(0, (i * 7) % (n + 1)))) for i in range(n)]

    def value(i, c):
        if i == c:
            return 4.0 * np.eye(3) + 0.1 * rng.standard_normal((3, 3))
        scale = 0.6 if abs(i - c) in (1, n - 1) else 0.01
        return scale * (np.eye(3) + 0.3 * rng.standard_normal((3, 3)))

    A = _bsr(3, 3, rows, n, value)
    with pkg.BlockSolver(autotune=0, amg_coarse_size=8) as sol:
        sol.setup(A, _none(3, 1, n, 4), _none(1, 3, 4, n), _identity(1, 4))
        nl = sol.amg_levels(pkg.SCR_HIER_A)
        As = [sol.export(pkg.SCR_HIER_A, l, pkg.SCR_EXPORT_OPERATOR) for l in range(nl)]
        Ps = [to_csr(sol.export(pkg.SCR_HIER_A, l, pkg.SCR_EXPORT_PROLONGATOR)) for l in range(nl - 1)]
        aggs = [sol.export(pkg.SCR_HIER_A, l, pkg.SCR_EXPORT_AGGREGATES) for l in range(nl - 1)]
    widths = np.diff((abs(to_csr(_bsr(1, 1, rows, n, lambda i, c: 1.0)))
                      @ amg.tentative_prolongator(aggs[0].astype(np.int64), 1)).indptr)
    assert nl >= 2 and widths.min() < 60 and widths.max() > 68
    for l in range(nl - 1):
        M = to_csr(As[l])
        P, _ = amg.smoothed_prolongator(M, amg.tentative_prolongator(aggs[l].astype(np.int64), 3))
        P = amg.truncate_prolongator(P, 3, 0.3, 5)
        assert abs(Ps[l] - P).max() <= 1e-12 * abs(P).max()
        Ac = P.T @ M @ P
        assert abs(to_csr(As[l + 1]) - Ac).max() <= 1e-11 * abs(Ac).max()


def _one_level(D):
    """Block system whose Shat is D (A = I, no coupling)."""
    n = D.shape[0]
    return (_identity(3, 4), _none(3, 1, 4, n), _none(1, 3, n, 4),
            _bsr(1, 1, [np.flatnonzero(D[i]) for i in range(n)], n, lambda i, c: D[i, c]))


def _hadamard(n):
    H = np.ones((1, 1))
    while H.shape[0] < n:
        H = np.block([[H, H], [H, -H]])
    return H


@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 33, 128, 560, 700])
@pytest.mark.parametrize("kind", ["shift", "ties", "random"])
def test_dense_inverse_exchanges_rows(n, kind):
    """Zero leading pivots (a cyclic shift of powers of two, whose inverse is
    exact), columns of equal magnitudes (a Hadamard matrix, bordered by the
    identity) and random entries with a zero diagonal, from one row to more than
    shared memory holds: the residual of an explicit inverse, at most
    8 n eps cond(D) |b|."""
    rng = np.random.default_rng(n)
    if kind == "shift":
        D = np.diag(2.0 ** rng.integers(-6, 7, n))[:, (np.arange(n) + 1) % n]
    elif kind == "ties":
        D = np.eye(n)
        m = 2 ** (n.bit_length() - 1)
        D[:m, :m] = _hadamard(m)
    else:
        D = rng.standard_normal((n, n))
        if n > 1:
            np.fill_diagonal(D, 0.0)
    b = rng.standard_normal(n)
    with pkg.BlockSolver(amg_max_levels=1, autotune=0) as sol:
        sol.setup(*_one_level(D))
        x = sol.amg_apply(pkg.SCR_HIER_SHAT, _dev(b)).cpu().numpy()
    if kind == "shift":
        assert np.array_equal(D @ x, b)
    assert np.linalg.norm(D @ x - b) <= 8 * n * np.finfo(float).eps * np.linalg.cond(D) * np.linalg.norm(b)


@pytest.mark.parametrize("n", [2, 17, 560, 700])
def test_singular_coarsest_operator_is_rejected(n):
    """Two equal rows leave an exact zero pivot in the last step; the handle
    takes another system afterwards."""
    D = np.eye(n)
    D[n - 2:, n - 2:] = 1.0
    with pkg.BlockSolver(amg_max_levels=1, autotune=0) as sol:
        with pytest.raises(pkg.ScrError, match="singular"):
            sol.setup(*_one_level(D))
        sol.setup(*_one_level(np.eye(n)))
        x = sol.amg_apply(pkg.SCR_HIER_SHAT, _dev(np.arange(n) + 1.0)).cpu().numpy()
    assert np.array_equal(x, np.arange(n) + 1.0)


@pytest.mark.parametrize("long", [33, 129, 300])
def test_block_operator_and_schur_rows_longer_than_a_group(long):
    """Rows of A, B, C and D with 33, 129 and 300 blocks (a warp takes rows above
    32, or eight rounds of one-column blocks) among rows of four: calA x against
    the definition (a row sums 4 long products at most, each off by eps/2 of the
    absolute sum), S x_p with a tight inner solve against D - C A^{-1} B."""
    n, rng = 320, np.random.default_rng(long)

    def pattern(special):
        rows = [sorted({i} | set(rng.choice(n, 3, replace=False).tolist())) for i in range(n)]
        for i in special:
            rows[i] = sorted({i} | set(rng.choice(n, long - 1, replace=False).tolist()))
        return rows

    some = lambda r, c: (lambda i, j: 0.02 * rng.standard_normal((r, c)))
    A = _bsr(3, 3, pattern([5, 17, 319]), n, lambda i, c: (i == c) * 4.0 * np.eye(3) + some(3, 3)(i, c))
    B, C = _bsr(3, 1, pattern([6, 17]), n, some(3, 1)), _bsr(1, 3, pattern([0, 7, 8]), n, some(1, 3))
    D = _bsr(1, 1, pattern([7, 318]), n, lambda i, c: (i == c) * 4.0 + some(1, 1)(i, c))
    from oracle.sparse import BlockOperator
    op = BlockOperator(A, B, C, D)
    x, xp = rng.standard_normal(4 * n), rng.standard_normal(n)
    with pkg.BlockSolver(autotune=0, rtol_I=1e-13, max_I=500, restart_inner=60) as sol:
        sol.setup(A, B, C, D)
        y = sol.apply_op(_dev(x)).cpu().numpy()
        yp = sol.apply_schur(_dev(xp)).cpu().numpy()
    K = op.full().tocsr()
    assert np.all(np.abs(y - K @ x) <= 4 * long * 1.2e-16 * (abs(K) @ np.abs(x)))
    Ad = to_csr(A).toarray()
    ref = to_csr(D) @ xp - to_csr(C) @ np.linalg.solve(Ad, to_csr(B) @ xp)
    assert np.linalg.norm(yp - ref) <= 1e-10 * np.linalg.norm(ref)
