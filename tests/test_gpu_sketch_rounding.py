"""The tensor-core sketches' rounding of A to the sketch precision, value by
value, and the dense-row kernel's chunks, several to a CTA."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu
FORMATS = {"fp16": (11, -14), "bf16": (8, -126), "fp32": (24, -126)}   # significand bits, least exponent


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_18411_gb300 import build
    build.build()
    from paper_2606_18411_gb300 import mrcqr as M
    return torch, M


def _round(x, prec):
    p, emin = FORMATS[prec]
    ex = np.maximum(np.frexp(x)[1] - 1, emin) - (p - 1)
    return np.ldexp(np.rint(np.ldexp(x, -ex)), ex)


def _values():
    out = [0.0, -0.0, 5e-324, -2.0 ** -1022, 1.0 - 2.0 ** -53]
    for t in (0, 1, 5, 13, 26, 27, 28, 36, 37, 38, 60, 120, 138, 139, 140):
        for f in (1.0, 1 + 2.0 ** -11, 1 + 2.0 ** -11 + 2.0 ** -52, 1 + 3 * 2.0 ** -11, -(1 + 2.0 ** -8),
                  1 + 2.0 ** -24, 1 + 3 * 2.0 ** -24, 2 - 2.0 ** -52):
            if abs(f) * 2.0 ** -t <= 1.0:
                out.append(f * 2.0 ** -t)
    return np.array(out)


# Row k = 0 of the transform is all ones: a column +B, -B, x with B its largest
# entry sums to the rounded x.  x sits in another K step of the tensor core than
# +B and -B, so the sum is exact.
@pytest.mark.parametrize("prec", ["fp16", "bf16", "fp32"])
@pytest.mark.parametrize("variant,m,rows", [(2, 512, (192, 193, 212)), (2, 511, (448, 449, 468)),
                                            (4, 2048, (0, 32, 640))])
@pytest.mark.parametrize("log2b", [0, -70, 90])
def test_rounding_of_each_value(env, prec, variant, m, rows, log2b):
    torch, M = env
    x = np.ldexp(_values(), log2b)
    n, B = len(x), 2.0 ** log2b
    s = min(m, 1024)
    seed = next(k for k in range(100) if 0 in O.sample_rows(m, s, k))
    d, idx = O.rademacher(m, seed), O.sample_rows(m, s, seed)
    A = np.zeros((m, n))
    A[rows[0]], A[rows[1]], A[rows[2]] = d[rows[0]] * B, -d[rows[1]] * B, d[rows[2]] * x
    Y = M.sketch(M.to_colmajor(A), s, prec, seed=seed, variant=variant).cpu().numpy()
    assert M.last_sketch_variant() == variant
    y = Y[int(np.flatnonzero(idx == 0)[0])] / (np.sqrt(2.0 / s) * np.sqrt(0.5))
    e = 13 - log2b                                     # the column's scale: its largest entry into [2^13, 2^14)
    want = _round(np.ldexp(_round(np.ldexp(x, e), prec), -e), "fp32")   # the sums are in FP32, without the scale
    # FP32 in two TF32 parts of 11 bits; tensor-core and FP32 subnormals may be zero
    tol = (2.0 ** -21 if prec == "fp32" else 2.0 ** -50) * np.abs(want) + 2.0 ** (-126 - e + 1)
    assert (np.abs(y - want) <= tol).all()


@pytest.mark.parametrize("m,n,s,ld", [(99968, 33, 66, 0), (70001, 130, 260, 70001), (1 << 17, 64, 128, 0),
                                      (200, 3, 6, 0)])
def test_dense_rows_over_chunks(env, m, n, s, ld):
    torch, M = env
    rng = np.random.default_rng(m)
    rows = np.unique(np.concatenate([rng.integers(0, m, 60), [0, m - 1]]))   # few nonzeros: a lost chunk shows
    A = np.zeros((m, n))
    A[rows] = rng.standard_normal((len(rows), n))
    Y = M.sketch(M.to_colmajor(A, ld=ld or None), s, "fp32", seed=9, variant=2).cpu().numpy()
    assert M.last_sketch_variant() == 2
    idx, d = O.sample_rows(m, s, 9), O.rademacher(m, 9)
    F = np.stack([(O.dct_row(int(k), m) / O.dct_coefficient(int(k), m))[rows] for k in idx])
    coef = (np.sqrt(2.0 / s) * np.where(idx == 0, np.sqrt(0.5), 1.0))[:, None]
    ref = coef * (F @ (d[rows, None] * A[rows]))
    # two TF32 parts (2^-21), FP32 twiddles of a few ulp, FP32 sums
    assert (np.abs(Y - ref) <= coef * 2.0 ** -18 * np.abs(A).sum(axis=0)[None, :]).all()


# FP32 sums run over at most 64 rows of a short matrix: 64 odd 18-bit integers add up exactly in FP32 (24 bits), 128
# of them to an odd sum above 2^24 do not.  Row k = 0 of the transform is all ones; variant 1: SIMT, 2: tensor cores.
@pytest.mark.parametrize("variant", [1, 2])
@pytest.mark.parametrize("m,s", [(384, 384), (1000, 600), (4096, 300)])   # m / 64 chunks at most 608 / (s / 64)
def test_short_matrices_keep_fp32_sums_of_64_rows(env, variant, m, s):
    torch, M = env
    n = 5
    seed = next(k for k in range(200) if 0 in O.sample_rows(m, s, k))
    d, idx = O.rademacher(m, seed), O.sample_rows(m, s, seed)
    X = (np.random.default_rng(m).integers(2 ** 16, 2 ** 17, (m, n)) * 2 + 1).astype(np.float64)
    X[::128] -= 1.0                                   # an even term in every 128 rows: their sum is odd
    Y = M.sketch(M.to_colmajor(d[:, None] * X), s, "fp32", seed=seed, variant=variant).cpu().numpy()
    assert M.last_sketch_variant() == variant
    want = np.sqrt(2.0 / s) * np.sqrt(0.5) * X.sum(axis=0)
    assert (np.abs(Y[int(np.flatnonzero(idx == 0)[0])] - want) <= 2.0 ** -50 * want).all()
