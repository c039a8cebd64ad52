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
