"""The SVD of the sketch (one-sided Jacobi from an orthogonal start) against LAPACK over its row counts:
below and above the orthogonal start, odd row and block counts, each register shape, graded, clustered
and rank-deficient rows."""
import numpy as np
import pytest
import torch

from paper_2203_07329_gb300 import tikhonov as tk

pytestmark = pytest.mark.gpu


def _rows(s, n, kind, gen):
    if kind == "graded":  # the sketch of an exponential spectrum
        Y = torch.randn(s, n, dtype=torch.float64, generator=gen) * torch.exp(-torch.arange(n) / (n / 18.0))
    elif kind == "flat":
        Y = torch.randn(s, n, dtype=torch.float64, generator=gen)
    elif kind == "deficient":  # rank s / 2, two equal rows, a zero row
        Y = torch.randn(s, s // 2, dtype=torch.float64, generator=gen) @ torch.randn(s // 2, n, dtype=torch.float64,
                                                                                     generator=gen)
        Y[1] = Y[0]
        Y[2] = 0.0
    else:  # "near": rows equal to 1e-9, which Y Y^T cannot tell apart in float64
        Y = torch.ones(s, 1, dtype=torch.float64) @ torch.randn(1, n, dtype=torch.float64, generator=gen)
        Y = Y + 1e-9 * torch.randn(s, n, dtype=torch.float64, generator=gen)
    return Y


# Singular values: an orthogonal transformation of Y moves them by a few s units of sigma_1 (normwise
# backward error, 2^-53 sqrt(s n) sigma_1 with a factor 8 for the rotations); V orthonormal on the
# nonzero ones to 1e-13 and Y V = U Sigma with orthogonal columns.
@pytest.mark.parametrize("s,n,kind", [(1, 5, "flat"), (2, 2, "flat"), (3, 7, "graded"), (63, 80, "graded"),
                                      (64, 64, "flat"), (65, 513, "graded"), (97, 130, "deficient"),
                                      (130, 1025, "graded"), (66, 2049, "flat"), (70, 4100, "graded"),
                                      (67, 100, "near"), (334, 700, "graded")])
def test_svd_matches_lapack(s, n, kind):
    gen = torch.Generator().manual_seed(100 * s + n)
    Y = _rows(s, n, kind, gen)
    sig, V, sweeps = tk.tk_sketch_svd(Y.cuda())
    sig, V, Yh = sig.cpu().numpy(), V.cpu().numpy(), Y.numpy()
    ref = np.linalg.svd(Yh, compute_uv=False)
    u = 2.0 ** -53 * ref[0] * np.sqrt(s * n)
    assert sweeps < 60
    assert np.max(np.abs(sig - ref)) <= 8 * u
    live = sig > 1e3 * u
    G = V[:, live].T @ V[:, live]
    assert np.max(np.abs(G - np.eye(G.shape[0]))) < 1e-13 * max(1.0, np.sqrt(s))
    # the right singular vectors: Y V has orthogonal columns of norm sigma, to the normwise error
    B = Yh @ V[:, live]
    assert np.max(np.abs(np.linalg.norm(B, axis=0) - sig[live])) <= 16 * u
    C = B.T @ B
    np.fill_diagonal(C, 0.0)
    assert np.max(np.abs(C)) <= 16 * u * ref[0]
