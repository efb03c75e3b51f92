"""W = A R^{-1} where its fast path needs care: panels that keep the substitution
at a ragged edge, columns of very different size.  References are correctly rounded products
(``oracle.product_rounded``) and the solve in FP64 arithmetic."""
import numpy as np
import pytest

from oracle import mrcqr_oracle as O

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2606_18411_gb300 import mrcqr as M
    return torch, M


def _triangle(n, rng):
    return np.triu(rng.standard_normal((n, n)) * 0.3) + np.diag(1.0 + rng.random(n))


def _column_residuals(A, W, R):
    """||A_j - (W R)_j|| against ||(|W| |R|)_j|| per column, over at most 32000 entries."""
    rows = np.arange(A.shape[0])[::max(1, A.size // 32000)]
    A, W = A[rows], W[rows]
    res = np.linalg.norm(A - O.product_rounded(W, R), axis=0)
    return res, np.linalg.norm(np.abs(W) @ np.abs(R), axis=0)


# A tiny diagonal entry just before the last column: the last panel, of 2, 8, 18 and 31 columns, would amplify and
# keeps the substitution, whose triangle ends at column n.
@pytest.mark.parametrize("n", [34, 40, 50, 63, 512 - 1])
def test_ragged_last_panel_keeps_its_substitution(env, n):
    torch, M = env
    rng = np.random.default_rng(n)
    R = _triangle(n, rng)
    R[n - 2, n - 2] = 1e-9
    A = rng.standard_normal((200, n))
    W = M.trsm(M.to_colmajor(A), M.to_colmajor(R)).cpu().numpy()
    assert np.isfinite(W).all()
    res, scale = _column_residuals(A, W, R)
    assert (res <= 4 * n * U * scale).all(), float((res / scale).max())


# R's first 32 rows 2^1200 above the others: zeros of W in those columns say nothing about the rows' size.
@pytest.mark.parametrize("n", [33, 64, 130])
def test_zeros_do_not_raise_a_row_reference(env, n):
    torch, M = env
    rng = np.random.default_rng(n)
    R = _triangle(n, rng)
    R[:32, :32] *= 2.0 ** 600
    R[:, 32:] *= 2.0 ** -600
    A = rng.standard_normal((150, n))
    A[:, :32] *= 2.0 ** 600
    A[:, 32:] *= 2.0 ** -600
    A[::2, :32] = 0.0
    W = M.trsm(M.to_colmajor(A), M.to_colmajor(R)).cpu().numpy()
    assert (W[::2, :32] == 0.0).all()
    res, scale = _column_residuals(A[::2, 32:] * 2.0 ** 600, W[::2, 32:], R[32:, 32:] * 2.0 ** 600)
    assert (res <= 4 * n * U * scale).all(), float((res / scale).max())


def _scales(n, order, span, rng):
    """Column scales over `span` (a power of two exponent for "random2"), in the given order."""
    if order == "random2":                            # 2^-span .. 2^span
        return 2.0 ** rng.integers(-span, span + 1, n)
    d = span ** (-np.arange(n) / max(n - 1, 1))
    return {"descending": d, "ascending": d[::-1], "random": rng.permutation(d)}[order]


SCALINGS = [("random", 1e6), ("random", 1e12), ("random", 1e18), ("descending", 1e18), ("ascending", 1e18),
            ("random2", 200)]


# Columns of A of very different size.  R = R_0 diag(d) with R_0 of unit columns, as a factor of A has it: equilibrated
# columns make every column's backward error that of a triangular solve.
@pytest.mark.parametrize("order,span", SCALINGS)
@pytest.mark.parametrize("n", [16, 32, 33, 64, 160, 512])
def test_trsm_columns_of_different_size(env, n, order, span):
    torch, M = env
    rng = np.random.default_rng(n)
    m = 2 * n + 131
    G = rng.standard_normal((m, n))
    d = _scales(n, order, span, rng)
    A, R = G * d, np.linalg.qr(G)[1] * d
    for fp64_products in (0, 1):
        W = M.trsm(M.to_colmajor(A), M.to_colmajor(R), fp64_products=fp64_products).cpu().numpy()
        # powers of two do not round, other scales enter A and R with one rounding: compare what was solved
        e = np.frexp(d)[1]
        res, scale = _column_residuals(np.ldexp(A, -e), W, np.ldexp(R, -e))
        assert (res <= 4 * n * U * scale).all(), (fp64_products, float((res / scale).max()))


@pytest.mark.parametrize("prec", ["bf16", "fp16", "fp32", "fp64", "auto"])
@pytest.mark.parametrize("order,span", [("random", 1e18), ("descending", 1e12), ("random2", 60)])
def test_factorization_of_columns_of_different_size(env, prec, order, span):
    torch, M = env
    rng = np.random.default_rng(5)
    m, n = 3000, 70
    d = _scales(n, order, span, rng)
    G = rng.standard_normal((m, n))
    A = G * d
    if prec == "auto":
        from paper_2606_18411_gb300 import selector
        selector.load_into_library()
    Q, R = (t.cpu().numpy() for t in M.factor(M.to_colmajor(A), prec=prec, seed=3))
    assert M.last_status()["status"] == "OK"
    e = np.frexp(d)[1]
    _check_factors(np.ldexp(A, -e), Q, np.ldexp(R, -e))


def _check_factors(A, Q, R):
    n = A.shape[1]
    assert np.linalg.norm(Q.T @ Q - np.eye(n)) <= 1e-13
    res, scale = _column_residuals(A, Q, R)
    # two triangular products and the Gram of well-conditioned columns
    assert (res <= 16 * n * U * scale).all(), float((res / scale).max())


def test_batched_plan_and_cholqr2_of_columns_of_different_size(env):
    torch, M = env
    rng = np.random.default_rng(11)
    shapes = [(700, 20), (900, 64), (1500, 150)]
    ds = [_scales(n, "random", 1e15, rng) for _, n in shapes]
    As = [rng.standard_normal(sh) * d for sh, d in zip(shapes, ds)]
    Ad = [M.to_colmajor(A) for A in As]
    Qs = [M.empty_colmajor(*sh) for sh in shapes]
    Rs = [M.empty_colmajor(sh[1], sh[1]) for sh in shapes]
    status = torch.zeros(len(shapes), dtype=torch.int32, device="cuda")
    M.BatchedPlan(Ad, Qs, Rs, ["fp16", "fp32", "fp64"], [1, 2, 3], status).execute()
    assert status.cpu().tolist() == [0, 0, 0]
    for A, d, Q, R in zip(As, ds, Qs, Rs):
        e = np.frexp(d)[1]
        _check_factors(np.ldexp(A, -e), Q.cpu().numpy(), np.ldexp(R.cpu().numpy(), -e))
    for A, d, Adev in zip(As, ds, Ad):
        Q, R = M.cholqr2(Adev)
        assert M.last_status()["status"] == "OK"
        e = np.frexp(d)[1]
        _check_factors(np.ldexp(A, -e), Q.cpu().numpy(), np.ldexp(R.cpu().numpy(), -e))


# R that is no factor of A: its columns say nothing about A's.  Columns of A graded over 1e25 against the identity, a
# triangle of its own, and a first block so ill-conditioned that W's columns differ by 1e12.
@pytest.mark.parametrize("kind", ["identity", "triangle", "ill_block"])
@pytest.mark.parametrize("m,n", [(300, 2), (130, 32), (257, 70), (400, 160)])
def test_trsm_with_an_unrelated_triangle(env, m, n, kind):
    torch, M = env
    rng = np.random.default_rng(m + n)
    A = rng.standard_normal((m, n)) * _scales(n, "random" if kind != "ill_block" else "ascending", 1e25, rng)
    R = np.eye(n) if kind == "identity" else np.linalg.qr(rng.standard_normal((2 * n, n)))[1]
    if kind == "ill_block":
        A = rng.standard_normal((m, n))
        k = min(32, n // 2)
        R[:k, k:] = 0.0
        R[:k, :k] *= (1e-12 ** (np.arange(k) / max(k - 1, 1)))[:, None]
    A[m // 2:m // 2 + 3] *= 1e-30                     # rows of another size keep their own references
    W = M.trsm(M.to_colmajor(A), M.to_colmajor(R)).cpu().numpy()
    if kind == "identity":
        np.testing.assert_array_equal(W, A)
    d = 2.0 ** -np.frexp(np.abs(A).max(0))[1]         # exact: keeps the reference's products in range
    res, scale = _column_residuals(A * d, W, R * d)
    assert (res <= 4 * n * U * scale).all(), float((res / scale).max())


# A non-finite entry in either half of a panel, in the first panel or with W to its left: the columns before it are
# those of the row without it.
@pytest.mark.parametrize("value", [np.inf, np.nan])
@pytest.mark.parametrize("col", [0, 5, 17, 40, 56, 69])
def test_nonfinite_entry_reaches_only_the_columns_after_it(env, col, value):
    torch, M = env
    rng = np.random.default_rng(col)
    m, n, row = 300, 70, 133
    R = _triangle(n, rng)
    A = rng.standard_normal((m, n))
    clean = M.trsm(M.to_colmajor(A), M.to_colmajor(R)).cpu().numpy()
    A[row, col] = value
    W = M.trsm(M.to_colmajor(A), M.to_colmajor(R)).cpu().numpy()
    np.testing.assert_array_equal(np.delete(W, row, 0), np.delete(clean, row, 0))
    assert not np.isfinite(W[row, col:]).any()
    # two solutions with backward errors gamma_n |W| |R|: apart by at most that through |R^-1|
    bound = 8 * n * U * (np.abs(clean[row]) @ np.abs(R)) @ np.abs(np.linalg.inv(R))
    assert (np.abs(W[row, :col] - clean[row, :col]) <= bound[:col]).all()


# A column of A that is zero in a row block: W there is what the columns before it make it, here 2^-40 of them.
@pytest.mark.parametrize("m,n,j", [(1, 20, 10), (150, 64, 31), (300, 70, 68)])
def test_trsm_zero_column_of_a(env, m, n, j):
    torch, M = env
    rng = np.random.default_rng(n)
    A = rng.standard_normal((m, n))
    A[:128, j] = 0.0
    A[128:, j] *= 2.0 ** -40
    R = np.eye(n)
    R[:j, j] = rng.standard_normal(j) * 2.0 ** -40
    W = M.trsm(M.to_colmajor(A), M.to_colmajor(R)).cpu().numpy()
    res, scale = _column_residuals(A, W, R)
    assert (res <= 4 * n * U * scale).all(), float((res / scale).max())
