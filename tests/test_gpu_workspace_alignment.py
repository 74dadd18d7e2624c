"""A caller's workspace at any address: the same results as from an aligned one."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2203_07329_gb300 import datagen, tikhonov as tk

pytestmark = pytest.mark.gpu


def _work(size, shift):
    return torch.empty(size + 256, dtype=torch.uint8, device="cuda")[shift:shift + size]


# order 700: panels of 256 rows, block rows and the levels of the inverse; 90: a single block row
@pytest.mark.parametrize("shift", [0, 8, 16, 40])
@pytest.mark.parametrize("precision", [tk.TK_PREC_FP64, tk.TK_PREC_MIXED])
@pytest.mark.parametrize("m,n", [(3000, 700), (1000, 90)])
def test_solve(m, n, precision, shift):
    p = datagen.make_ridge_problem(m, n, datagen.spectrum("log", n, hi=1.0, lo=1e-3),
                                   datagen.log_lambdas(3, 1e-4, 1e-1), seed=n)
    A, b, lams = p.A.cuda(), p.b.cuda(), p.lambdas.numpy()
    o = tk.opts_default(precision=precision, s=min(4 * n, m))
    r0 = tk.tk_solve(A, b, lams, o)
    r = tk.tk_solve(A, b, lams, o, work=_work(tk.workspace_size(tk.make_problem(A, b), 3, o), shift))
    assert r.status == tk.TK_OK
    assert float((r.X - r0.X).norm()) <= 1e-10 * float(r0.X.norm())


@pytest.mark.parametrize("shift", [8, 16])
def test_lcurve(shift):
    m, n, N, Nr = 2000, 150, 6, 3
    p = datagen.make_ridge_problem(m, n, datagen.spectrum("log", n, hi=1.0, lo=1e-3),
                                   datagen.log_lambdas(N, 1e-6, 1e-1), seed=n)
    A, b, lams = p.A.cuda(), p.b.cuda(), p.lambdas.numpy()
    o = tk.opts_default(precision=tk.TK_PREC_MIXED, s=4 * n)
    X0, _, c0 = tk.tk_lcurve(A, b, lams, Nr, o)
    X, _, c = tk.tk_lcurve(A, b, lams, Nr, o, work=_work(tk.lcurve_workspace_size(A, b, N, Nr, o), shift))
    assert c == c0
    assert float((X - X0).norm()) <= 1e-10 * float(X0.norm())


@pytest.mark.parametrize("shift", [8, 16])
def test_cholesky(shift):
    n = 400
    Y = torch.randn(3 * n, n, dtype=torch.float64, generator=torch.Generator().manual_seed(1)).cuda()
    Cm = Y.T @ Y
    R0, _ = tk.tk_cholesky_shifted(Cm, [1e-3, 1.0], emulate=True)
    lam, R = np.array([1e-3, 1.0]), torch.empty_like(R0)
    w = _work(tk.lib().tk_cholesky_emulated_workspace(n, 2), shift)
    st = tk.lib().tk_cholesky_shifted_emulated(C.c_void_p(Cm.data_ptr()), n, lam.ctypes.data_as(C.c_void_p), 2,
                                               C.c_void_p(R.data_ptr()), None, C.c_void_p(w.data_ptr()), w.numel(), None)
    assert st == tk.TK_OK
    assert torch.equal(R, R0)
