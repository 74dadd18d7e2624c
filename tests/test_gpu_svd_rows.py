"""The SVD of the sketch at the ends of its range: rows longer than the registers of a block pair hold, rows that
depend on each other exactly, and rows far from unit scale."""
import numpy as np
import pytest
import torch

from paper_2203_07329_gb300 import tikhonov as tk

pytestmark = pytest.mark.gpu


def _check(Y, max_sweeps):
    s, n = Y.shape
    sig, V, sweeps = tk.tk_sketch_svd(torch.from_numpy(Y).cuda())
    sig, V = sig.cpu().numpy(), V.cpu().numpy()
    ref = np.linalg.svd(Y, compute_uv=False)
    # the normwise error of an orthogonal transformation, as for the other shapes of this call
    u = 2.0 ** -53 * ref[0] * np.sqrt(s * n)
    assert np.max(np.abs(sig - ref)) <= 8 * u
    live = sig > 1e3 * u
    G = V[:, live].T @ V[:, live]
    assert np.max(np.abs(G - np.eye(G.shape[0]))) < 1e-13 * max(1.0, np.sqrt(s))
    B = (Y / ref[0]) @ V[:, live]
    assert np.max(np.abs(np.linalg.norm(B, axis=0) - sig[live] / ref[0])) <= 16 * u / ref[0]
    assert sweeps < max_sweeps


# 8192 values are the most that a block pair holds in registers; rows beyond are rotated in memory.  3, 5: fewer
# rows than two blocks; 66 and 70: from the orthogonal start, an odd and an even number of blocks
@pytest.mark.parametrize("s,n", [(3, 8192), (5, 8193), (70, 8192), (66, 8193), (6, 20001), (67, 20011)])
def test_long_rows(s, n):
    gen = np.random.default_rng(s + n)
    _check(gen.standard_normal((s, n)) * np.exp(-np.arange(n) / (n / 6.0)), 30)


# rows that depend on each other exactly (fewer nonzero columns than rows, equal columns, equal rows), below and
# above the 64 rows of the orthogonal start: each sweep leaves rounding errors of the sweep before, which end as
# zero rows and not as pairs that are rotated for ever (80 sweeps is the cap)
def _dependent(kind):
    gen = np.random.default_rng(7)
    if kind == "ones":
        return np.ones((30, 40))
    if kind == "outer":
        return np.outer(gen.standard_normal(8), gen.standard_normal(40))
    s, r, n = {"zero columns 16": (16, 6, 36), "zero columns 32": (32, 20, 50), "zero columns 96": (96, 40, 100),
               "equal columns 40": (40, 5, 50), "equal columns 80": (80, 30, 90)}[kind]
    X = gen.standard_normal((s, r))
    return np.tile(X, (1, n // r)) if kind.startswith("equal") else np.hstack([X, np.zeros((s, n - r))])


@pytest.mark.parametrize("kind", ["ones", "outer", "zero columns 16", "zero columns 32", "zero columns 96",
                                  "equal columns 40", "equal columns 80"])
def test_dependent_rows(kind):
    _check(_dependent(kind), 30)


# powers of two on the whole matrix: the squares and fourth powers of a row norm leave float64's range long before
# the norm does
@pytest.mark.parametrize("e", [-400, -330, -270, 270, 330, 400])
@pytest.mark.parametrize("s,n", [(20, 30), (80, 130)])
def test_scales(s, n, e):
    gen = np.random.default_rng(s)
    _check(np.ldexp(gen.standard_normal((s, n)), e), 30)


# more rows than the orthogonal start takes (no row of s values fits in shared memory): rows that are orthogonal from
# the start, so that one sweep ends it
def test_more_rows_than_the_orthogonal_start_takes():
    s = 25602
    d = torch.exp(-torch.arange(s, dtype=torch.float64) / 3000.0)
    sig, V, sweeps = tk.tk_sketch_svd(torch.diag(d).cuda())
    assert sweeps == 1
    assert float((sig.cpu() - d).abs().max()) <= 2.0 ** -50
    V -= torch.eye(s, dtype=torch.float64, device="cuda")
    assert float(V.abs().max()) <= 2.0 ** -50
