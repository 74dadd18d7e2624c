"""The measured work of the library: what its users have it do, over the range of sizes they bring.

A case is one call of tk_solve, tk_solve_batched or tk_lcurve on data shaped like the paper's
synthetic matrices (Section 4): A = U diag(sigma) V^T, x_true with standard normal entries,
b = A x_true + 1e-3 N(0, 1), lambdas log-spaced.  Here U is an m x min(m, n) Gaussian matrix over
sqrt(m) (its columns orthonormal up to a few per cent) and V a random-sign cosine transform
(exactly orthogonal), so that the inputs are made in milliseconds on the GPU instead of by a QR.
"""
import math

import numpy as np
import torch

from paper_2203_07329_gb300 import tikhonov as tk

SKETCH = {"srht": tk.TK_SKETCH_SRHT, "gauss": tk.TK_SKETCH_GAUSS, "sparse": tk.TK_SKETCH_SPARSE,
          "srdct": tk.TK_SKETCH_SRDCT}
PRECISION = {"fp64": tk.TK_PREC_FP64, "mixed": tk.TK_PREC_MIXED}
PRECOND = {"chol": tk.TK_PRECOND_CHOL, "lowrank": tk.TK_PRECOND_LOWRANK}


def _case(kind="solve", *, m, n, N, dtype="f64", precision="fp64", precond="chol", sketch="srht", over=4,
          spectrum="log", lo=1e-6, tau=200.0, lam_lo=1e-6, lam_hi=1.0, pad=0, count=1, N_refine=0, name=None):
    """kind: solve, batch or lcurve.  m, n: rows and columns (of the largest problem of a batch).
    N lambdas in lam_lo..lam_hi.  over: sketch rows per unit of min(m, n); 0 = twice the statistical
    dimension (low rank).  spectrum: log (1..lo) or exp (exp(-i / tau)).  pad: columns between n and
    the row stride of A.  count: problems of a batch.  N_refine: second-sweep lambdas of an L-curve."""
    c = dict(kind=kind, m=m, n=n, N=N, dtype=dtype, precision=precision, precond=precond, sketch=sketch, over=over,
             spectrum=spectrum, lo=lo, tau=tau, lam_lo=lam_lo, lam_hi=lam_hi, pad=pad, count=count,
             N_refine=N_refine)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small fit with a known lambda: the least a caller asks for, all launches and latency
        _case(m=2000, n=64, N=1, sketch="gauss", lam_lo=1e-2, lam_hi=1e-2, name="one_lambda_2000x64_fp64"),
        # the small workload of the benchmark, in the default precision ...
        _case(m=4096, n=256, N=8, sketch="gauss", name="small_4096x256_fp64"),
        # ... and in the mixed form
        _case(m=4096, n=256, N=8, sketch="gauss", precision="mixed", name="small_4096x256_mixed"),
        # an ordinary fit in the default precision and options (float64, SRHT, s = 4n)
        _case(m=65536, n=1024, N=16, name="ordinary_65536x1024_fp64"),
        # float32 data with odd sizes and a padded row stride, sparse embedding (s = 16n), mixed form
        _case(m=50021, n=777, N=11, dtype="f32", precision="mixed", sketch="sparse", over=16, lo=1e-5, lam_lo=1e-5,
              pad=3, name="ragged_50021x777_f32_mixed"),
        # the headline workload of the benchmark: a large float64 A, 32 lambdas, mixed form
        _case(m=262144, n=2048, N=32, precision="mixed", lo=1e-8, lam_lo=1e-8, name="large_262144x2048_mixed"),
        # the precision form (float32 A, BF16 Gaussian sketch s = 2n, 64 lambdas), a quarter of its rows
        _case(m=262144, n=4096, N=64, dtype="f32", precision="mixed", sketch="gauss", over=2, lo=1e-5, lam_lo=1e-5,
              name="precision_262144x4096_f32_mixed"),
        # underdetermined (Algorithm 2), exponential spectrum
        _case(m=1024, n=65536, N=16, spectrum="exp", lam_hi=1e-1, name="under_1024x65536_fp64"),
        # a small statistical dimension: Algorithm 3, sketch size 2 sd, default precision
        _case(m=30000, n=1000, N=16, precond="lowrank", sketch="gauss", over=0, spectrum="exp", tau=50.0,
              lam_lo=1e-4, name="lowrank_30000x1000_fp64"),
        # serving: uneven independent problems in one call, every other one low rank
        _case("batch", m=65536, n=1024, N=16, dtype="f32", precision="mixed", sketch="gauss", lo=1e-5, tau=50.0,
              count=16, name="uneven_batch_16_f32_mixed"),
        # the L-curve (Section 4.3): a coarse sweep, then a second one around its corner
        _case("lcurve", m=65536, n=1024, N=24, N_refine=8, precision="mixed", lo=1e-8, lam_lo=1e-8,
              name="lcurve_65536x1024_mixed"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp64", "mixed", "mixed", "mixed", "under", "lowrank", "batch", "lcurve"])
    lam_lo = 10.0 ** rng.uniform(-6, -2)
    dtype = rng.choice(["f64", "f32"])
    sketch = rng.choice(["srht", "gauss", "srht", "sparse", "srdct"])
    over = 16 if sketch == "sparse" else rng.choice([3, 4, 5])
    pad = rng.choice([0, 0, rng.randint(1, 7)])
    if kind in ("fp64", "lowrank"):
        m = _log_uniform(rng, 2000, 65536)
        n = min(_log_uniform(rng, 48, 1024), m // 6)
        N = rng.randint(1, 16)
        if kind == "lowrank":
            return _case(m=m, n=n, N=N, precond="lowrank", sketch="gauss", over=0, spectrum="exp",
                         tau=rng.uniform(n / 25, n / 15), lam_lo=max(lam_lo, 1e-4), pad=pad)
        return _case(m=m, n=n, N=N, sketch=sketch, over=over, lam_lo=lam_lo, lo=1e-6, pad=pad)
    if kind == "mixed":
        m = _log_uniform(rng, 4000, 262144)
        n = min(_log_uniform(rng, 64, 2048), m // 6)
        return _case(m=m, n=n, N=rng.randint(2, 40), dtype=dtype, precision="mixed", sketch=sketch, over=over,
                     lam_lo=lam_lo, lo=1e-5 if dtype == "f32" else 1e-6, pad=pad)
    if kind == "under":
        n = _log_uniform(rng, 2000, 65536)
        m = min(_log_uniform(rng, 48, 1024), n // 6)
        return _case(m=m, n=n, N=rng.randint(1, 16), sketch=sketch, over=over, spectrum="exp", tau=m / 5.0,
                     lam_lo=lam_lo, lam_hi=1e-1, pad=pad)
    if kind == "batch":
        m = _log_uniform(rng, 4000, 40000)
        return _case("batch", m=m, n=min(_log_uniform(rng, 80, 700), m // 6), N=rng.randint(2, 16), dtype=dtype,
                     precision="mixed", sketch="gauss", lo=1e-5, tau=50.0, lam_lo=lam_lo, count=rng.randint(3, 12),
                     pad=pad)
    m = _log_uniform(rng, 4000, 65536)
    precision = rng.choice(["mixed", "fp64"]) if m < 20000 else "mixed"
    return _case("lcurve", m=m, n=min(_log_uniform(rng, 64, 1024), m // 6), N=rng.randint(12, 24),
                 N_refine=rng.randint(0, 8), dtype=dtype if precision == "mixed" else "f64", precision=precision,
                 sketch=rng.choice(["srht", "gauss"]), lo=1e-6, lam_lo=1e-7, pad=pad)


def _sizes(case):
    """(m, n, low rank) of every problem of the case: a batch has uneven ones, the first the largest."""
    if case["kind"] != "batch":
        return [(case["m"], case["n"], case["precond"] == "lowrank")]
    out = []
    for p in range(case["count"]):
        f, g = (p * 0.6180339887498949) % 1.0, (p * 0.7548776662466927) % 1.0
        n = max(32, int(case["n"] * (1.0 - 0.93 * f)))
        out.append((max(4 * n, 2000, int(case["m"] * (1.0 - 0.95 * g))), n, p % 2 == 1))
    return out


def _sigma(case, k, lowrank):
    i = torch.arange(k, dtype=torch.float64)
    if case["spectrum"] == "exp" or (case["kind"] == "batch" and lowrank):
        return torch.exp(-i / case["tau"])
    return torch.pow(torch.tensor(case["lo"], dtype=torch.float64), i / max(k - 1, 1))


def _lambdas(case):
    return np.geomspace(case["lam_lo"], case["lam_hi"], case["N"]) if case["N"] > 1 else np.array([case["lam_hi"]])


def _sketch_rows(case, m, n, lowrank):
    c = min(m, n)
    if lowrank:
        sd = float((1.0 / (1.0 + case["lam_lo"] / _sigma(case, c, True) ** 2)).sum())
        return min(c, 2 * math.ceil(sd))
    return min((case["over"] or 4) * c, max(m, n))


def _rows_cosine(T, sign):
    """Rows of T (in place) times diag(sign) times the orthonormal DCT-II of their length."""
    r, k = T.shape
    T.mul_(sign)
    f = torch.fft.fft(torch.cat([T[:, ::2], T[:, 1::2].flip(1)], dim=1))
    w = torch.exp(-0.5j * math.pi * torch.arange(k, device=T.device, dtype=torch.float64) / k).to(f.dtype)
    T.copy_((f * w).real.mul_(math.sqrt(2.0 / k)))
    T[:, 0] *= math.sqrt(0.5)


def _problem(case, m, n, lowrank, gen):
    """One A (m x n view with row stride n + pad) and b."""
    dt = torch.float64 if case["dtype"] == "f64" else torch.float32
    c, L = min(m, n), max(m, n)
    sig = _sigma(case, c, lowrank).to("cuda", dt)
    G = torch.empty((L, c + (case["pad"] if m >= n else 0)), dtype=dt, device="cuda")
    sign = torch.randint(0, 2, (2, c), generator=gen, device="cuda").to(dt) * 2 - 1
    step = max(1, (1 << 26) // c)
    for r0 in range(0, L, step):
        T = torch.randn((min(step, L - r0), c), generator=gen, dtype=dt, device="cuda")
        T.mul_(sig / math.sqrt(L))
        for k in range(2):
            _rows_cosine(T, sign[k])
        G[r0:r0 + step, :c] = T
    if m >= n:
        A = G[:, :n]
    else:
        A = torch.empty((m, n + case["pad"]), dtype=dt, device="cuda")[:, :n]
        A.copy_(G.T)
    x = torch.randn(n, generator=gen, dtype=torch.float64, device="cuda")
    b = torch.randn(m, generator=gen, dtype=torch.float64, device="cuda") * 1e-3
    step = max(1, (1 << 26) // n)
    for r0 in range(0, m, step):
        b[r0:r0 + step] += A[r0:r0 + step].to(torch.float64) @ x
    return A, b


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return [_problem(case, m, n, lr, gen) for m, n, lr in _sizes(case)]


def prepare(case, seed):
    pairs = _inputs(case, seed)
    opts = [tk.opts_default(sketch=SKETCH[case["sketch"]], s=_sketch_rows(case, m, n, lr), seed=int(seed) % 1000 + 1,
                            precision=PRECISION[case["precision"]],
                            precond=tk.TK_PRECOND_LOWRANK if lr else tk.TK_PRECOND_CHOL)
            for m, n, lr in _sizes(case)]
    lam = _lambdas(case)
    if case["kind"] == "batch":
        need = tk.workspace_size_batched(pairs, case["N"], opts)
    elif case["kind"] == "lcurve":
        need = tk.lcurve_workspace_size(*pairs[0], case["N"], case["N_refine"], opts[0])
    else:
        need = tk.workspace_size(tk.make_problem(*pairs[0]), case["N"], opts[0])
    # the caller's workspace, kept for every solve of the same shapes
    return dict(case=case, pairs=pairs, opts=opts, lam=lam,
                work=torch.empty(need, dtype=torch.uint8, device="cuda"))


def run(state):
    case, pairs, opts, lam, work = (state[k] for k in ("case", "pairs", "opts", "lam", "work"))
    if case["kind"] == "batch":
        Xs, _, _ = tk.tk_solve_batched(pairs, np.tile(lam, (len(pairs), 1)), opts, work=work)
        return Xs
    A, b = pairs[0]
    if case["kind"] == "lcurve":
        X, pts, _ = tk.tk_lcurve(A, b, lam, case["N_refine"], opts[0], work=work)
        return {"X": X, **{k: np.array([p[k] for p in pts]) for k in ("lam", "rnorm", "xnorm")}}
    return tk.tk_solve(A, b, lam, opts[0], work=work).X


def work(case):
    """Bytes: A and b read once, X written once.  Flops: the sketch, the Gram matrix (or, low rank, the
    products of an s x n SVD), a factorization per lambda, and per lambda the two products with A of the
    LSQR iterations that Section 3.1.2 expects for ten digits (contraction sqrt(c / s) per step)."""
    nbytes = flops = 0.0
    N = case["N"] + case["N_refine"]
    for m, n, lr in _sizes(case):
        c, L = min(m, n), max(m, n)
        s = _sketch_rows(case, m, n, lr)
        steps = math.log(1e10) / math.log(math.sqrt(2.0 if lr else max(s / c, 1.5)))
        nbytes += (8 if case["dtype"] == "f64" else 4) * m * n + 8 * m + 8 * N * n
        flops += (2.0 * s if case["sketch"] == "gauss" else math.log2(L)) * m * n
        flops += 4.0 * s * s * c if lr else s * c * c + N * c ** 3 / 3.0
        flops += N * steps * 4.0 * m * n
    return {"bytes": nbytes, "flops": flops}


def _gram64(A, b):
    """A^T A and A^T b in float64, by blocks of rows."""
    m, n = A.shape
    C = torch.zeros((n, n), dtype=torch.float64, device=A.device)
    g = torch.zeros(n, dtype=torch.float64, device=A.device)
    step = max(1, (1 << 27) // n)
    for r0 in range(0, m, step):
        T = A[r0:r0 + step].to(torch.float64)
        C += T.T @ T
        g += T.T @ b[r0:r0 + step]
    return C, g


def _ridge64(A, b, lams):
    """x_lambda for every lambda: the R factor of [A b] and a QR of [R; sqrt(lambda) I] per lambda where
    lambda is small, else normal equations (A A^T where m < n) with refinement against A itself."""
    m, n = A.shape
    if m < n:
        A64 = A.to(torch.float64)
        C, out = A64 @ A64.T, []
        eye = torch.eye(m, dtype=torch.float64, device=A.device)
        for lam in lams:
            L = torch.linalg.cholesky(C + lam * eye)
            z = torch.zeros((m, 1), dtype=torch.float64, device=A.device)
            for _ in range(4):
                z += torch.cholesky_solve(b[:, None] - A64 @ (A64.T @ z) - lam * z, L)
            out.append((A64.T @ z)[:, 0])
        return torch.stack(out)
    eye = torch.eye(n, dtype=torch.float64, device=A.device)
    if min(lams) < 1e-6:
        R = torch.linalg.qr(torch.cat([A.to(torch.float64), b[:, None]], dim=1), mode="r").R
        c = torch.cat([R[:n, n:], torch.zeros((n, 1), dtype=torch.float64, device=A.device)])
        out = []
        for lam in lams:
            S = torch.linalg.qr(torch.cat([torch.cat([R[:n, :n], math.sqrt(lam) * eye]), c], dim=1), mode="r").R
            out.append(torch.linalg.solve_triangular(S[:n, :n], S[:n, n:], upper=True)[:, 0])
        return torch.stack(out)
    C, g0 = _gram64(A, b)
    Ls = [torch.linalg.cholesky(C + lam * eye) for lam in lams]
    X = torch.stack([torch.cholesky_solve(g0[:, None], L)[:, 0] for L in Ls])
    lam_t = torch.tensor(np.asarray(lams), device=A.device)[:, None]
    step = max(1, (1 << 26) // n)
    for _ in range(2):
        G = -lam_t * X
        for r0 in range(0, m, step):
            T = A[r0:r0 + step].to(torch.float64)
            G += (b[None, r0:r0 + step] - X @ T.T) @ T
        X += torch.stack([torch.cholesky_solve(G[i][:, None], L)[:, 0] for i, L in enumerate(Ls)])
    return X


def _norms64(A, b, X):
    r2 = torch.zeros(X.shape[0], dtype=torch.float64, device=A.device)
    step = max(1, (1 << 26) // A.shape[1])
    for r0 in range(0, A.shape[0], step):
        r2 += (b[None, r0:r0 + step] - X @ A[r0:r0 + step].to(torch.float64).T).square().sum(1)
    return r2.sqrt().cpu().numpy(), X.square().sum(1).sqrt().cpu().numpy()


def _corner(lam, rn, xn):
    """Index of the largest curvature of (ln rn, ln xn) over ln lam, three-point differences."""
    t, P, Q = np.log(lam), np.log(rn), np.log(xn)
    best, at = 0.0, 1
    for k in range(1, len(t) - 1):
        h1, h2 = t[k] - t[k - 1], t[k + 1] - t[k]
        d = [(-h2 / h1 * F[k - 1] + (h2 / h1 - h1 / h2) * F[k] + h1 / h2 * F[k + 1]) / (h1 + h2) for F in (P, Q)]
        dd = [2 * (F[k - 1] / h1 - (1 / h1 + 1 / h2) * F[k] + F[k + 1] / h2) / (h1 + h2) for F in (P, Q)]
        kappa = (d[0] * dd[1] - dd[0] * d[1]) / (d[0] ** 2 + d[1] ** 2) ** 1.5
        if k == 1 or kappa > best:
            best, at = kappa, k
    return at


def exact(case, seed):
    pairs, lam = _inputs(case, seed), _lambdas(case)
    if case["kind"] == "batch":
        return [_ridge64(A, b, lam) for A, b in pairs]
    A, b = pairs[0]
    X = _ridge64(A, b, lam)
    if case["kind"] != "lcurve":
        return X
    rn, xn = _norms64(A, b, X)
    k = _corner(lam, rn, xn)
    q = case["N_refine"]
    more = np.exp(np.linspace(math.log(lam[k - 1]), math.log(lam[k + 1]), q + 2)[1:-1])
    if q:
        X = torch.cat([X, _ridge64(A, b, more)])
        rn2, xn2 = _norms64(A, b, X[len(lam):])
        lam, rn, xn = np.concatenate([lam, more]), np.concatenate([rn, rn2]), np.concatenate([xn, xn2])
        at = np.argsort(lam, kind="stable")
        X, lam, rn, xn = X[torch.from_numpy(at).to(X.device)], lam[at], rn[at], xn[at]
    return {"X": X, "lam": lam, "rnorm": rn, "xnorm": xn}
