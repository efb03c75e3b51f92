"""W = A R^{-1} where its fast path needs care: panels that keep the substitution
at a ragged edge.  References are correctly rounded products
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
    """||A_j - (W R)_j|| against ||(|W| |R|)_j|| per column."""
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
