"""The row-block products W = A R^{-1} and Q = W X and the slicing they share
with the Gram, at the edges of their tiles and of their fast paths.  The
references are correctly rounded products (``oracle.product_rounded``)."""
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


def _triangle(n, kind, rng):
    R = np.triu(rng.standard_normal((n, n)) * 0.3) + np.diag(1.0 + rng.random(n))
    if kind == "tiny_diagonal":   # panels whose inverse would amplify: they keep the substitution
        for k in {n // 3, n - 2}:
            R[k, k] = 1e-7
    elif kind == "negative":
        R *= np.where(np.arange(n) % 2, -1.0, 1.0)[:, None]
    elif kind == "wide_range":    # rows over 2^-120 .. 1: row scalings beyond the fast slicing's range
        R *= 2.0 ** (-120.0 * np.arange(n) / max(n - 1, 1))[:, None]
    return R


# one column, around one panel (32), around the four panels of one exact accumulation (128), the widest;
# rows below, at and above a block (128); odd leading dimensions of A and W
@pytest.mark.parametrize("m,n,kind", [(1, 1, "plain"), (127, 31, "plain"), (128, 32, "tiny_diagonal"),
                                      (129, 33, "negative"), (300, 64, "wide_range"), (257, 96, "tiny_diagonal"),
                                      (140, 128, "plain"), (140, 129, "tiny_diagonal"), (131, 161, "wide_range"),
                                      (129, 512, "tiny_diagonal")])
def test_trsm_residual_at_panel_edges(env, m, n, kind):
    torch, M = env
    rng = np.random.default_rng(1000 * m + n)
    R = _triangle(n, kind, rng)
    A = rng.standard_normal((m, n))
    A[:, 0] = 0.0                                     # zeros take the general slicing
    W = M.trsm(M.to_colmajor(A, ld=m + 1 + m % 2), M.to_colmajor(R)).cpu().numpy()
    assert np.isfinite(W).all()
    res = np.linalg.norm(A - O.product_rounded(W, R))
    # backward error of a triangular solve: gamma_n || |W| |R| ||
    assert res <= 4 * n * U * np.linalg.norm(np.abs(W) @ np.abs(R))


def test_trsm_nonfinite_stays_in_its_rows_and_columns(env):
    torch, M = env
    rng = np.random.default_rng(7)
    m, n = 300, 70
    R = _triangle(n, "plain", rng)
    A = rng.standard_normal((m, n))
    clean = M.trsm(M.to_colmajor(A), M.to_colmajor(R)).cpu().numpy()
    A[5, 40] = np.inf
    W = M.trsm(M.to_colmajor(A), M.to_colmajor(R)).cpu().numpy()
    np.testing.assert_array_equal(W[:, :32], clean[:, :32])       # panels before the entry
    np.testing.assert_array_equal(np.delete(W, 5, 0), np.delete(clean, 5, 0))
    assert not np.isfinite(W[5, 40:]).any()


@pytest.mark.parametrize("m,n,ld", [(1, 1, 0), (130, 32, 131), (127, 33, 0), (200, 129, 0), (129, 160, 131)])
def test_finalize_within_bound_at_tile_edges(env, m, n, ld):
    torch, M = env
    rng = np.random.default_rng(m + 10 * n)
    W = rng.standard_normal((m, n))
    W[::3] *= 2.0 ** -45                              # whole rows: each row has its own reference
    W[:, ::4] *= 2.0 ** -40                           # columns below the fast slicing's range
    X = np.triu(rng.standard_normal((n, n)))
    Q = M.finalize_q(M.to_colmajor(W, ld=ld or None), M.to_colmajor(X)).cpu().numpy()
    exact = O.product_rounded(W, X)
    bound = 2 * U * np.abs(exact) + 2.0 ** -57 * n * np.abs(W).max(1)[:, None] * np.abs(X).max(0)[None, :]
    assert np.all(np.abs(Q - exact) <= bound)


# Level sums beyond 2^22: every balanced digit of 0x3F7F7F7F7F800000 / 2^62 after the first is -128, so 128 equal
# rows make the largest sums there are, and the readout has to correct them with conversions.
@pytest.mark.parametrize("m,n", [(128, 3), (4096, 40), (1000, 130)])
def test_largest_level_sums(env, m, n):
    torch, M = env
    x = float(0x3F7F7F7F7F800000) / 2.0 ** 62
    W = np.full((m, n), x)
    W[:, 1::2] *= -1.0
    G = M.gram(M.to_colmajor(W)).cpu().numpy()
    exact = O.product_rounded(np.ascontiguousarray(W.T), W)
    upper = np.triu(np.ones((n, n), bool))
    assert np.all(np.abs(G - exact)[upper] <= 2 * U * np.abs(exact)[upper] + 2.0 ** -57 * m * x * x)
    X = np.triu(np.full((n, n), x))
    Q = M.finalize_q(M.to_colmajor(W), M.to_colmajor(X)).cpu().numpy()
    ref = O.product_rounded(W, X)
    assert np.all(np.abs(Q - ref) <= 2 * U * np.abs(ref) + 2.0 ** -57 * n * x * x)


@pytest.mark.parametrize("m,n,ld", [(31, 5, 32), (33, 64, 33), (65, 65, 66), (4000, 70, 4001), (600, 192, 600)])
def test_gram_quads_at_edges(env, m, n, ld):
    torch, M = env
    rng = np.random.default_rng(m + n)
    W = rng.standard_normal((m, n))
    W[rng.random((m, n)) < 0.2] = 0.0                 # zeros
    W[rng.random((m, n)) < 0.1] *= 2.0 ** -50         # far below the column's reference
    G = M.gram(M.to_colmajor(W, ld=ld)).cpu().numpy()
    exact = O.product_rounded(np.ascontiguousarray(W.T), W)
    C = np.abs(W).max(0)
    upper = np.triu(np.ones((n, n), bool))
    assert np.all(np.abs(G - exact)[upper] <= (2 * U * np.abs(exact) + 2.0 ** -57 * m * C[:, None] * C[None, :])[upper])


# The 64-column tiles of wide W: at and around their widths (161, 192, 256, 289, 512 take them, 160, 224 and 257 do
# not), heights around a block of 128 rows, an odd leading dimension; a non-finite entry stays in its row.
@pytest.mark.parametrize("m,n,ld", [(129, 160, 0), (127, 161, 128), (257, 192, 0), (130, 224, 131), (131, 256, 0),
                                    (128, 257, 0), (200, 289, 0), (1, 320, 0), (150, 512, 151)])
def test_finalize_of_wide_matrices(env, m, n, ld):
    torch, M = env
    rng = np.random.default_rng(m + n)
    W = rng.standard_normal((m, n))
    W[::3] *= 2.0 ** -45                              # each row has its own reference
    W[:, ::4] *= 2.0 ** -40                           # columns below the fast slicing's range
    W[rng.random((m, n)) < 0.05] = 0.0
    X = np.triu(rng.standard_normal((n, n)))
    Q = M.finalize_q(M.to_colmajor(W, ld=ld or None), M.to_colmajor(X)).cpu().numpy()
    rows = np.arange(m)[::max(1, m * n // 16000)]
    exact = O.product_rounded(W, X, rows=rows)
    bound = 2 * U * np.abs(exact) + 2.0 ** -57 * n * np.abs(W[rows]).max(1)[:, None] * np.abs(X).max(0)[None, :]
    assert np.all(np.abs(Q[rows] - exact) <= bound)
    W[m // 2, n // 3] = np.nan
    Qn = M.finalize_q(M.to_colmajor(W), M.to_colmajor(X)).cpu().numpy()
    np.testing.assert_array_equal(np.delete(Qn, m // 2, 0), np.delete(Q, m // 2, 0))
    assert np.isnan(Qn[m // 2]).all()


def test_batched_wide_problems_match_single_launches(env):
    torch, M = env
    rng = np.random.default_rng(4)
    shapes = [(900, 161), (700, 64), (1300, 320), (640, 224)]
    As = [M.to_colmajor(rng.standard_normal(sh)) for sh in shapes]
    out = []
    for per_problem in (0, 1):
        Qs, Rs = [M.empty_colmajor(*sh) for sh in shapes], [M.empty_colmajor(sh[1], sh[1]) for sh in shapes]
        status = torch.full((len(shapes),), -1, dtype=torch.int32, device="cuda")
        M.BatchedPlan(As, Qs, Rs, ["fp32"] * 4, [1, 2, 3, 4], status, oz_per_problem=per_problem).execute()
        assert status.cpu().tolist() == [0] * 4
        out.append([t.cpu().numpy() for t in Qs + Rs])
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
