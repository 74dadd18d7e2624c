"""The float64 form from digits on matrices that no scaling of rows and columns evens out: as close to the oracle's
solution as on the float64 pipe.  The digits of an entry are relative to its row's and its column's largest, so they
perturb column j by 2^-55 of its largest entry: the error of a float64 QR of A, not of each entry."""
import numpy as np
import pytest
import torch

import oracle
from paper_2203_07329_gb300 import tikhonov as tk

pytestmark = pytest.mark.gpu

M, N = 2400, 240


def _graded(kind, rng):
    A = rng.standard_normal((M, N))
    if kind.startswith("outliers"):
        big = rng.random((M, N)) < 0.01
        if kind == "outliers but for 5 columns":
            big[:, :5] = False
        A[big] *= 1e8
    elif kind == "one outlier":
        A[7, 3] *= 1e10
    elif kind == "every entry":
        A *= 10.0 ** (-10 * rng.random((M, N)))
    elif kind == "rows and columns":
        A *= 10.0 ** (-8 * rng.random((M, 1))) * 10.0 ** (-8 * rng.random((1, N)))
    else:  # two blocks of full size, the other two 1e-9 of it
        A[:, 100:] *= 1e-9
        A[1200:, :100] *= 1e-9
    return A


# errors within a factor of 2 of the pipe's and 64 float64 units, in the norm of x and in that of its contributions to
# A x (each x_j times the norm of its column)
@pytest.mark.parametrize("kind", ["outliers", "outliers but for 5 columns", "one outlier", "every entry",
                                  "rows and columns", "blocks"])
@pytest.mark.parametrize("shift", [1e-8, 1e-12])
def test_as_close_as_the_float64_pipe(kind, shift):
    rng = np.random.default_rng(17)
    A = _graded(kind, rng)
    b = A @ (rng.standard_normal(N) / np.abs(A).max(0)) + 1e-3 * rng.standard_normal(M)
    lam = shift * np.linalg.norm(A, 2) ** 2
    ref = oracle.ref_ridge_qr(A, b, lam, refine=3)
    col = np.linalg.norm(A, axis=0)
    err = {}
    for emulate in (1, 0):
        r = tk.tk_solve(torch.from_numpy(A).cuda(), torch.from_numpy(b).cuda(), [lam],
                        tk.opts_default(s=4 * N, sketch=tk.TK_SKETCH_GAUSS, emulate_fp64=emulate))
        assert r.status == tk.TK_OK
        d = r.X[0].cpu().numpy() - ref
        err[emulate] = (np.linalg.norm(d) / np.linalg.norm(ref), np.linalg.norm(d * col) / np.linalg.norm(ref * col))
    for e1, e0 in zip(err[1], err[0]):
        assert e1 <= 2 * e0 + 64 * 2.0 ** -53, err
