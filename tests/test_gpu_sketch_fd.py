"""The FP64 sketch as a four-step transform (variant 6) against dense sums of
the oracle's transform rows, at the edges of its tiles, ranges and classes."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_18411_gb300 import build
    build.build()
    from paper_2606_18411_gb300 import mrcqr as M
    return torch, M


def _check(Y, A, s, seed):
    m = A.shape[0]
    idx, d = O.sample_rows(m, s, seed), O.rademacher(m, seed)
    F = np.stack([O.dct_row(int(k), m) / O.dct_coefficient(int(k), m) for k in idx])
    coef = (np.sqrt(2.0 / s) * np.where(idx == 0, np.sqrt(0.5), 1.0))[:, None]
    X = d[:, None] * A
    ref = coef * (F.astype(np.longdouble) @ X.astype(np.longdouble)).astype(np.float64)
    # FP64 cosines in the reference (2^-53 each, products and sums in at least 64 bits); first-step sums off by 2^-52 of
    # the column maximum C, 2^-50 C per term of the m / 16 of the second step; two roundings of the result
    C = np.abs(A).max(axis=0)[None, :]
    bound = coef * (2.0 ** -52 * np.abs(A).sum(axis=0)[None, :] + 2.0 ** -53 * m * C) + 3 * U * np.abs(ref)
    assert np.all(np.abs(Y - ref) <= bound)
    return ref


# one column and one past a column block; fewer samples than classes x 32 and more; J = m / 32 at and off the
# 128-row blocks; odd leading dimensions; columns of very different size, zeros, a zero column
@pytest.mark.parametrize("m,n,s,ld", [(1 << 15, 1, 160, 0), (32 * 1025, 3, 161, 32 * 1025 + 1), (1 << 16, 129, 258, 0),
                                      (32 * 1151, 5, 700, 0), (1 << 15, 2, 4096, 0)])
def test_four_step_sketch_against_dense(env, m, n, s, ld):
    torch, M = env
    rng = np.random.default_rng(m + n)
    A = rng.standard_normal((m, n)) * 2.0 ** rng.integers(-200, 200, (1, n))
    A[rng.random((m, n)) < 0.1] = 0.0
    A[::7] *= 2.0 ** -36
    if n > 2:
        A[:, 1] = 0.0
    Ad = M.to_colmajor(A, ld=ld or None)
    Y = M.sketch(Ad, s, "fp64", seed=5, variant=6).cpu().numpy()
    assert M.last_sketch_variant() == 6
    cols = np.arange(n) if n < 10 else np.array([0, 1, 63, 127, 128])
    _check(Y[:, cols], A[:, cols], s, 5)
    assert np.array_equal(Y, M.sketch(Ad, s, "fp64", seed=5).cpu().numpy())     # the automatic choice here


def test_four_step_sketch_all_ones_and_nonfinite(env):
    torch, M = env
    m, n, s = 1 << 15, 3, 192
    A = np.ones((m, n))
    A[:, 2] = 1.0 - 2.0 ** -53                        # the largest significand: the largest first-step sums
    _check(M.sketch(M.to_colmajor(A), s, "fp64", seed=8, variant=6).cpu().numpy(), A, s, 8)
    A[100, 1] = np.nan
    Y = M.sketch(M.to_colmajor(A), s, "fp64", seed=8, variant=6).cpu().numpy()
    assert np.isnan(Y[:, 1]).all() and np.isfinite(Y[:, [0, 2]]).all()


@pytest.mark.parametrize("ldq", [0, 3 * (1 << 15)])
def test_factorization_takes_it_with_q_as_scratch(env, ldq):
    torch, M = env
    from paper_2606_18411_gb300 import inputs
    m, n = 1 << 15, 96
    A = inputs.make_matrix(m, n, 1e14, seed=3)
    Q = M.empty_colmajor(m, n, ld=ldq or None)
    R = M.empty_colmajor(n, n)
    M.factor_ex(M.to_colmajor(A), Q, R, prec="fp64", seed=4, escalate=False)
    st = M.last_status()
    assert M.last_sketch_variant() == 6 and st["status"] == "OK" and st["ortho_fro"] <= 1e-13
    assert O.residual_error(A, Q[:m].cpu().numpy(), R.cpu().numpy())[0] <= 1e-13


# Q as the leading rows of a taller array: the FP64 sketch's scratch leaves the rows between its columns alone, in
# the columns of Q (the four-step form, 6, even ldq) or in the workspace (odd ldq; digit planes, 5).  Q and R are
# those of a packed Q bit for bit.
@pytest.mark.parametrize("m,n,pad,variant", [(1 << 15, 96, 2, 6), (1 << 15, 80, 1, 6), (9000, 100, 64, 5),
                                             (4099, 30, 1, 5), (1 << 15, 1, 6, 5), (32 * 2048, 128, 128, 6)])
def test_rows_between_the_columns_of_q_are_kept(env, m, n, pad, variant):
    torch, M = env
    from paper_2606_18411_gb300 import inputs
    A = M.to_colmajor(inputs.make_matrix(m, n, 1e10 if n > 1 else 1.0, seed=m + n))
    outs = []
    for ld in (m, m + pad):
        full = torch.full((n, ld), 7.25, dtype=torch.float64, device="cuda")
        Q, R = full.t()[:m], M.empty_colmajor(n, n)
        M.factor_ex(A, Q, R, prec="fp64", seed=4, escalate=False)
        assert M.last_status()["status"] == "OK" and M.last_sketch_variant() == variant
        assert bool((full[:, m:] == 7.25).all())
        outs.append((Q.cpu().numpy(), R.cpu().numpy()))
    np.testing.assert_array_equal(outs[0][0], outs[1][0])
    np.testing.assert_array_equal(outs[0][1], outs[1][1])


def test_sizes_the_four_step_form_does_not_take(env):
    torch, M = env
    A = np.random.default_rng(1).standard_normal((1 << 15, 4))
    for m, s in ((1 << 15, 159), ((1 << 15) - 8, 200), (1 << 14, 200)):
        Y = M.sketch(M.to_colmajor(A[:m]), s, "fp64", seed=2, variant=6).cpu().numpy()
        assert M.last_sketch_variant() == 5
        _check(Y, A[:m], s, 2)


def _sketch_time(torch, M, m, n, s):
    A = torch.randn((n, m), dtype=torch.float64, device="cuda").t()
    M.sketch(A, s, "fp64", seed=1)
    assert M.last_sketch_variant() == 6
    t = []
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        M.sketch(A, s, "fp64", seed=1)
        b.record()
        b.synchronize()
        t.append(a.elapsed_time(b))
    return sorted(t)[len(t) // 2]


# Heights off the multiples of 4096 cost what their rows cost: 5% fewer rows than 2^20 take at most a quarter more
# (ragged last blocks, one more range), not twice the time.
def test_time_follows_the_rows(env):
    torch, M = env
    assert _sketch_time(torch, M, 1000000, 128, 256) <= 1.25 * _sketch_time(torch, M, 1 << 20, 128, 256)
