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


def _hard_square_roots():
    """d whose square roots lie closest to the middle of two doubles: p = N / 2^53, N odd, N^2 = k mod 2^e for small k."""
    out = []
    for e in (54, 55):                                # d in [1, 2) and in [2, 4)
        M = 1 << e
        for k in range(-2047, 2048, 8):               # k = 1 mod 8 has four roots
            x = 1
            for b in range(3, e):
                if ((x * x - k) >> b) & 1:
                    x += 1 << (b - 1)
            for r in (x, -x, x + M // 2, M // 2 - x):
                for N in {r % M, r % M + M}:
                    D = (N * N - k) >> e
                    if 1 << 53 <= N < 1 << 54 and 1 << 52 <= D < 1 << 53:
                        out.append(np.ldexp(float(D), e - 106))
    return out


def test_pivot_is_correctly_rounded(env):
    torch, M = env
    from paper_2606_18411_gb300 import _lib
    rng = np.random.default_rng(1)
    one = 1.0 + np.arange(2000) * 2.0 ** -52
    ones = 2.0 - (1 + np.arange(2000)) * 2.0 ** -52   # the last significands below 2, all ones first
    d = np.concatenate([np.ldexp(1.0 + rng.random(400000), rng.integers(-1022, 1023, 400000)), _hard_square_roots(),
                        one, one ** 2, ones, 2 * ones, ones ** 2, np.nextafter(ones ** 2, 4.0),
                        [2.0 ** -1022, np.finfo(np.float64).max, 5e-324, 2.0 ** -1023, 1e-310]])
    bad = np.array([0.0, -0.0, -1.0, -5e-324, np.inf, -np.inf, np.nan])
    dev = torch.from_numpy(np.concatenate([d, bad])).cuda()
    p, y = torch.empty_like(dev), torch.empty_like(dev)
    assert _lib.load().mrcqr_debug_pivot_sqrt(dev.numel(), dev.data_ptr(), p.data_ptr(), y.data_ptr(), None) == 0
    torch.cuda.synchronize()
    p, y = p.cpu().numpy(), y.cpu().numpy()
    np.testing.assert_array_equal(p[:len(d)], np.sqrt(d))          # IEEE square root and division
    np.testing.assert_array_equal(y[:len(d)], 1.0 / np.sqrt(d))
    assert (p[len(d):] == -1.0).all() and (y[len(d):] == -1.0).all()


@pytest.mark.parametrize("n", [87, 88, 89, 96, 97])   # one CTA up to 88, panels of 32 beyond
def test_cholesky_at_the_switch(env, n):
    test_cholesky_sizes(env, n)
