"""The one-CTA Cholesky and the sketch QR of the preconditioner at the edges of
their forms: the triangle in shared memory (n <= 160) and blocked beyond, the
one-launch QR and the panel QR in registers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2606_18411_gb300 import mrcqr as M
    return torch, M


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 128, 159, 160, 161, 193, 512])
def test_cholesky_sizes(env, n):
    torch, M = env
    rng = np.random.default_rng(n)
    m = 2 * n + 70
    A = rng.standard_normal((m, n))
    P = np.eye(n) + np.triu(rng.standard_normal((n, n)) * (0.3 / np.sqrt(n)), 1)   # a factor that is not diagonal
    Rs = np.linalg.qr(A)[1] @ P
    kappa = np.linalg.cond(P)
    Q, R = (t.cpu().numpy() for t in M.cholqr_precond(M.to_colmajor(A), M.to_colmajor(Rs)))
    assert M.last_status()["status"] == "OK"
    assert np.array_equal(R, np.triu(R)) and (np.diag(R) != 0).all()
    # Cholesky QR of W = A Rs^-1: ||Q^T Q - I|| <= c (m n + n (n + 1)) u kappa(W)^2 (Yamamoto et al. 2015), and the
    # backward errors of the two triangular products
    e = (m * n + n * (n + 1)) * U * kappa ** 2
    assert np.linalg.norm(Q.T @ Q - np.eye(n), 2) <= 6 * e
    assert np.linalg.norm(A - Q @ R) <= 8 * n * U * np.linalg.norm(np.abs(Q) @ np.abs(R)) * kappa


@pytest.mark.parametrize("n,j", [(40, 39), (130, 70), (200, 199), (200, 33)])
def test_cholesky_breakdown_is_reported(env, n, j):
    torch, M = env
    A = np.random.default_rng(n).standard_normal((3 * n, n))
    A[:, j] = 0.0                                     # an exactly zero pivot
    M.cholqr_precond(M.to_colmajor(A), M.to_colmajor(np.eye(n)))
    assert M.last_status()["status"] == "BREAKDOWN"


# around the panel width (8), one CTA against panels (n = 32 / 64), the rows a
# thread holds (128 per step), the smallest and the widest
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n,s", [(1, 1), (1, 200), (7, 14), (8, 127), (9, 128), (16, 129), (32, 64), (32, 512),
                                 (33, 66), (33, 255), (64, 128), (64, 400), (65, 130), (100, 256), (100, 257),
                                 (161, 513), (256, 512), (512, 1024), (40, 3000)])
def test_sketch_qr_sizes(env, prec, n, s):
    torch, M = env
    rng = np.random.default_rng(100 * n + s)
    Y = rng.standard_normal((s, n)) * 2.0 ** rng.integers(-8, 9, (1, n))
    if n > 8:
        Y[:, n // 2] = 0.0
    if prec == "fp32":
        Y = Y.astype(np.float32).astype(np.float64)
    R = M.sketch_qr(M.to_colmajor(Y), prec).cpu().numpy()
    assert np.isfinite(R).all() and np.array_equal(R, np.triu(R))
    # Householder QR: R^T R = (Y + E)^T (Y + E), |E_j| <= gamma(s n)|Y_j| per column; s sqrt(n) u covers it here
    g = 4 * s * np.sqrt(n) * (2.0 ** -24 if prec == "fp32" else U)
    c = np.linalg.norm(Y, axis=0)
    assert (np.abs(R.T @ R - Y.T @ Y) <= 2 * g * np.outer(c, c)).all()
