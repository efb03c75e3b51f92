"""What a user of this library has it do, as cases whose time and outputs can be compared between two
versions of the code: whole factorizations over the range of the paper's tables and of the repository's
benchmark, a batched plan, and the step-level calls that other methods are built from.

Matrices are A = G diag(sigma) V^T with G Gaussian (condition number 1 + O(sqrt(n/m))) and V Haar, the
spectrum geometric from 1 to 1/kappa (the paper's workload).  The thin Q of a matrix is determined by A in
FP64 only up to about kappa * 2^-53, whatever the method, so kappa stays where two correct methods still
agree to 1e-9 (well inside each precision's own regime); a pass costs the same at every kappa of a regime."""
import math

import numpy as np
import torch

from paper_2606_18411_gb300 import mrcqr as M

# condition number used with each sketch precision
KAPPA = {"bf16": 20.0, "fp16": 1e3, "fp32": 1e5, "fp64": 1e5, "auto": 1e5}
MAX_M, MAX_N = 1 << 20, 512


def listed():
    return [
        # one small system, as a Krylov method or a service meets it: launches and latency count
        _factor("small_n32", 4096, 32, "fp32"),
        # few columns, a short matrix, the cheapest sketch
        _factor("narrow_n16", 16384, 16, "bf16"),
        # the paper's stability experiment at its own shape with its own sketch (c = 3n real-FFT bins)
        _factor("stability_n50", 131072, 50, "fp32", s_factor=3, transform="rfft"),
        # the paper's timing table, m = 2^20, with the half-precision sketch
        _factor("table_n64_half", 1 << 20, 64, "fp16"),
        # a matrix as data give it, odd row count (no 16-byte alignment of the columns), precision left to the library
        _factor("ragged_n100_auto", 1000003, 100, "auto"),
        # the paper's timing table, FP64 sketch (what an unknown condition number needs)
        _factor("table_n128_double", 1 << 20, 128, "fp64"),
        # the benchmark's wider problems
        _factor("wide_n256_single", 1 << 20, 256, "fp32"),
        _factor("widest_n512_double", 1 << 20, 512, "fp64"),
        # many uneven factorizations in one plan (block Krylov, randomized-SVD power steps)
        {"name": "batch_64", "kind": "batch", "count": 64, "lo": 1 << 14, "hi": 1 << 17},
        # the comparison method of the paper: two Cholesky-QR passes
        {"name": "cholqr2_n96", "kind": "cholqr2", "m": 1 << 18, "n": 96, "kappa": 1e3},
        # the preconditioning step alone: W = A R^-1
        {"name": "trsm_n320", "kind": "trsm", "m": 300001, "n": 320, "kappa": 1e5},
        # the FP64 sketch alone, c = 2n rows of the DCT
        {"name": "sketch_n160_double", "kind": "sketch", "m": 1 << 18, "n": 160, "c": 320},
    ]


def draw(rng):
    kind = rng.choice(["factor"] * 7 + ["batch", "cholqr2", "trsm", "sketch"])
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(8, 64), "lo": 1 << rng.randint(12, 14), "hi": 1 << rng.randint(15, 17)}
    n = _log_int(rng, 8, MAX_N)
    m = _log_int(rng, max(1 << 12, 8 * n), MAX_M)
    if kind == "factor":
        tf = rng.choice(["dct", "dct", "dct", "rfft"])
        c = _factor(None, m, n, rng.choice(["fp16", "bf16", "fp32", "fp64", "auto"]), rng.choice([2, 2, 3]), tf)
        del c["name"]
        return c
    if kind == "sketch":
        return {"kind": kind, "m": m, "n": n, "c": rng.choice([2, 3]) * n}
    return {"kind": kind, "m": m, "n": n, "kappa": 10.0 ** rng.uniform(1, 3 if kind == "cholqr2" else 5)}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _prepare_batch(case, seed)
    m, n = case["m"], case["n"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    B = _spectrum_rows(n, case.get("kappa", 1.0), gen)
    state = {"case": case, "seed": int(seed), "A": _matrix(m, B, gen)}
    if kind == "trsm":
        R = torch.linalg.qr(B, mode="r")[1]
        state["R"] = M.to_colmajor(torch.sign(torch.diagonal(R))[:, None] * R)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        state["plan"].execute()
        return state["q"], state["r"], state["status"]
    A, seed = state["A"], state["seed"]
    if kind == "factor":
        return M.factor(A, prec=case["prec"], seed=seed, s_factor=case["s_factor"], transform=case["transform"])
    if kind == "cholqr2":
        return M.cholqr2(A)
    if kind == "trsm":
        return M.trsm(A, state["R"])
    return M.sketch(A, case["c"], prec="fp64", seed=seed)


def work(case):
    """Bytes: inputs read once, outputs written once.  Operations: the method's own, at one per product and
    one per sum -- the triangular solve, the Gram, Q and the check at m n^2 each, a fast transform of A."""
    if case["kind"] == "batch":
        ps = _problems(case)
        return {"bytes": sum(8.0 * (2 * m * n + n * n) for m, n, _ in ps),
                "flops": sum(4.0 * m * n * n + 2.5 * m * n * math.log2(m) for m, n, _ in ps)}
    m, n, kind = case["m"], case["n"], case["kind"]
    if kind == "sketch":
        return {"bytes": 8.0 * (m + case["c"]) * n, "flops": 2.5 * m * n * math.log2(m)}
    if kind == "trsm":
        return {"bytes": 8.0 * (2 * m * n + n * n), "flops": 1.0 * m * n * n}
    if kind == "cholqr2":   # first pass: the Gram of A (a read of A); second pass: solve, Gram, Q, check
        return {"bytes": 8.0 * (2 * m * n + n * n), "flops": 5.0 * m * n * n}
    return {"bytes": 8.0 * (2 * m * n + n * n), "flops": 4.0 * m * n * n + 2.5 * m * n * math.log2(m)}


def exact(case, seed):
    """The same outputs from torch in FP64: Householder QR, a triangular solve, a fast cosine transform."""
    kind = case["kind"]
    if kind == "batch":
        q, r = [], []
        for m, n, A in _batch_matrices(case, seed):
            Q, R = _householder(A)
            q.append(Q.t().reshape(-1))
            r.append(R.t().reshape(-1))
        return torch.cat(q), torch.cat(r), None
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    B = _spectrum_rows(case["n"], case.get("kappa", 1.0), gen)
    A = _matrix(case["m"], B, gen)
    if kind == "trsm":
        R = torch.linalg.qr(B, mode="r")[1]
        R = torch.sign(torch.diagonal(R))[:, None] * R
        return torch.linalg.solve_triangular(R, A, upper=True, left=False)
    if kind == "sketch":
        return _dct_sketch(A, case["c"], seed)
    return _householder(A)


# --- inputs -------------------------------------------------------------------------------------------


def _factor(name, m, n, prec, s_factor=2, transform="dct"):
    return {"name": name, "kind": "factor", "m": m, "n": n, "prec": prec, "kappa": KAPPA[prec], "s_factor": s_factor,
            "transform": transform}


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _spectrum_rows(n, kappa, gen):
    """diag(sigma) V^T, n x n."""
    V = torch.linalg.qr(torch.randn((n, n), dtype=torch.float64, device="cuda", generator=gen))[0]
    sigma = kappa ** (-torch.arange(n, dtype=torch.float64, device="cuda") / max(n - 1, 1))
    return sigma[:, None] * V.t()


def _matrix(m, B, gen):
    """G B / sqrt(m), column-major m x n, G Gaussian."""
    G = torch.randn((B.shape[0], m), dtype=torch.float64, device="cuda", generator=gen)
    return (B.t() @ G).mul_(1.0 / math.sqrt(m)).t()


def _problems(case):
    """(m, n, precision) of every problem of a batch: sizes belong to the case, values to the seed."""
    rng = np.random.Generator(np.random.Philox(case["count"] + case["lo"] + case["hi"]))
    return [(int(rng.integers(case["lo"], case["hi"] + 1)), int(rng.choice([16, 32, 64, 128])),
             str(rng.choice(["fp16", "fp32", "fp64"]))) for _ in range(case["count"])]


def _batch_matrices(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    for m, n, prec in _problems(case):
        yield m, n, _matrix(m, _spectrum_rows(n, KAPPA[prec], gen), gen)


def _prepare_batch(case, seed):
    ps = _problems(case)
    q = torch.zeros(sum(m * n for m, n, _ in ps), dtype=torch.float64, device="cuda")
    r = torch.zeros(sum(n * n for _, n, _ in ps), dtype=torch.float64, device="cuda")
    As = [A for _, _, A in _batch_matrices(case, seed)]
    Qs, Rs, at, ar = [], [], 0, 0
    for m, n, _ in ps:
        Qs.append(q[at:at + m * n].view(n, m).t())
        Rs.append(r[ar:ar + n * n].view(n, n).t())
        at, ar = at + m * n, ar + n * n
    status = torch.zeros(len(ps), dtype=torch.int32, device="cuda")
    plan = M.BatchedPlan(As, Qs, Rs, [p for _, _, p in ps], [seed + i for i in range(len(ps))], status, use_graph=True)
    return {"case": case, "plan": plan, "q": q, "r": r, "status": status, "As": As}


# --- plain FP64 references ----------------------------------------------------------------------------


def _householder(A):
    Q, R = torch.linalg.qr(A)
    s = torch.sign(torch.diagonal(R))
    return Q * s, s[:, None] * R


def _philox_word0(c0, c1, key):
    """Word 0 of Philox4x32-10 (Salmon et al., SC'11) of the counters (c0, c1, 0, 0)."""
    sh, mask = np.uint64(32), np.uint64(0xFFFFFFFF)
    x = [np.asarray(c0, np.uint64), np.full_like(np.asarray(c0, np.uint64), c1), np.uint64(0), np.uint64(0)]
    k0, k1 = int(key) & 0xFFFFFFFF, (int(key) >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * x[0], np.uint64(0xCD9E8D57) * x[2]
        x = [(p1 >> sh) ^ x[1] ^ np.uint64(k0), p1 & mask, (p0 >> sh) ^ x[3] ^ np.uint64(k1), p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return x[0]


def _dct_sketch(A, c, seed):
    """sqrt(m/c) times c sampled rows of the orthonormal DCT-II of D A (even-extended FFT of length 2m)."""
    m, n = A.shape
    d = torch.from_numpy(1.0 - 2.0 * (_philox_word0(np.arange(m), 0, seed) & np.uint64(1)).astype(np.float64)).cuda()
    draws = (_philox_word0(np.arange(m - c, m), 1, seed) * (np.arange(m - c, m, dtype=np.uint64) + np.uint64(1))) >> np.uint64(32)
    picked = set()
    for j, t in zip(range(m - c, m), draws.tolist()):
        picked.add(t if t not in picked else j)
    k = torch.tensor(sorted(picked), dtype=torch.int64, device="cuda")
    turn = torch.exp(-1j * math.pi * k.to(torch.float64) / (2 * m))
    scale = math.sqrt(2.0 / c) * (1.0 - (1.0 - math.sqrt(0.5)) * (k == 0).to(torch.float64))
    Y = torch.empty((n, c), dtype=torch.float64, device="cuda")
    for j in range(n):
        x = A[:, j] * d
        f = torch.fft.fft(torch.cat([x, x.flip(0)]))[k]
        Y[j] = 0.5 * (turn * f).real * scale
    return Y.t()
