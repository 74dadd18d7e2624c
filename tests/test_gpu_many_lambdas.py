"""The float64 form with more lambdas than its digit routes take or keep an inverse of."""
import numpy as np
import pytest
import torch

from paper_2203_07329_gb300 import tikhonov as tk

pytestmark = pytest.mark.gpu


def _solve_exact(A, b, lam):
    n = A.shape[1]
    B = np.vstack([A, np.sqrt(lam) * np.eye(n)])
    return np.linalg.lstsq(B, np.concatenate([b, np.zeros(n)]), rcond=None)[0]


# more lambdas than one emulated Cholesky takes (8191): every lambda is solved, on the float64 pipe's Cholesky
@pytest.mark.parametrize("m,n,N", [(2000, 40, 8191), (2000, 40, 8193), (70, 1000, 8200)])
def test_many_lambdas(m, n, N):
    gen = np.random.default_rng(5)
    A = gen.standard_normal((m, n)) / np.sqrt(max(m, n))
    b = gen.standard_normal(m)
    lams = np.geomspace(1e-3, 1.0, N)
    r = tk.tk_solve(torch.from_numpy(A).cuda(), torch.from_numpy(b).cuda(), lams,
                    tk.opts_default(sketch=tk.TK_SKETCH_GAUSS, s=4 * min(m, n)))
    assert r.status == tk.TK_OK
    X = r.X.cpu().numpy()
    assert np.isfinite(X).all()
    for i in (0, 1, N // 2, 8190, N - 1):
        x = _solve_exact(A, b, lams[i])
        assert np.linalg.norm(X[i] - x) <= 1e-10 * np.linalg.norm(x)


# factors of order 512 and less are inverted explicitly however many lambdas there are (m >= n; beyond, the inverse of
# N c^2 > 8e7, or 2.7e8 from digits, makes way for substitution)
@pytest.mark.parametrize("c,N,emulate", [(200, 2100, 0), (300, 3200, 1)])
def test_small_factors_are_inverted(c, N, emulate):
    gen = np.random.default_rng(6)
    m = 4 * c
    A = torch.from_numpy(gen.standard_normal((m, c)) / np.sqrt(m)).cuda()
    b = torch.from_numpy(gen.standard_normal(m)).cuda()
    tk.tk_profile_collect()
    tk.tk_profile_enable(True)
    try:
        r = tk.tk_solve(A, b, np.geomspace(1e-2, 1.0, N), tk.opts_default(s=4 * c, emulate_fp64=emulate))
        ph = tk.tk_profile_collect()
    finally:
        tk.tk_profile_enable(False)
    assert r.status == tk.TK_OK
    assert ph["precond_inverse"]["launches"] == 1
