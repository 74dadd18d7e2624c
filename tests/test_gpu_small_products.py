"""The float32 products of at most 16 lambdas (pairs of lambdas per instruction)."""
import pytest
import torch

from paper_2203_07329_gb300 import datagen, tikhonov as tk

pytestmark = pytest.mark.gpu


# 1 .. 16 lambdas (odd counts: a half-empty pair), columns around the 4 of a lane, the 128 of a step and the
# 512 of a block, rows that leave groups of 4 and 8 incomplete, row strides with and without 16-byte rows.
# Refined to the float64 solution: each form within 1e-10 of the minimiser.
@pytest.mark.parametrize("m,n,N,pad", [(1003, 5, 1, 0), (1001, 130, 3, 2), (1030, 127, 4, 1), (4097, 513, 5, 3),
                                       (2050, 516, 8, 0), (1999, 200, 9, 1), (3001, 1027, 16, 1), (9, 6, 7, 0)])
def test_mixed_solve_of_few_lambdas(m, n, N, pad):
    p = datagen.make_ridge_problem(m, n, datagen.spectrum("log", n, hi=1.0, lo=1e-3),
                                   datagen.log_lambdas(N, 1e-4, 1e-1), seed=m + n)
    buf = torch.zeros(m, n + pad, dtype=torch.float64, device="cuda")
    buf[:, :n] = p.A.cuda()
    A, b, lams = buf[:, :n], p.b.cuda(), p.lambdas.numpy()
    kw = dict(sketch=tk.TK_SKETCH_GAUSS, s=min(2 * n, m))
    r1 = tk.tk_solve(A, b, lams, tk.opts_default(precision=tk.TK_PREC_MIXED, lsqr_tc=0, **kw))
    r0 = tk.tk_solve(A, b, lams, tk.opts_default(emulate_fp64=0, **kw))
    for i in range(N):
        assert float((r1.X[i] - r0.X[i]).norm() / r0.X[i].norm()) < 2e-10, lams[i]
