"""The grouped engine's product tiles: lambda classes of 4, 8, 16 and more, problems narrower and wider than a
column tile (512 or 1024), odd sizes and strides, the low-rank applies, against each problem solved on its own."""
import numpy as np
import pytest
import torch

from paper_2203_07329_gb300 import datagen, tikhonov as tk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 3, 7, 16, 21])
def test_grouped_tiles_match_single_solves(N):
    pairs, opts, lams = [], [], []
    for k, (m, n) in enumerate([(4103, 33), (2500, 130), (5001, 515), (9000, 64), (4400, 1031), (3001, 258)]):
        low = k % 2 == 1
        sig = datagen.spectrum("exp", n, tau=n / 12.0) if low else datagen.spectrum("log", n, hi=1.0, lo=1e-3)
        p = datagen.make_ridge_problem(m, n, sig, datagen.log_lambdas(N, 1e-3, 1.0), seed=m, dtype=torch.float32)
        pad = k % 3
        full = torch.full((m, n + pad), float("nan"), dtype=torch.float32, device="cuda")
        full[:, :n] = p.A.cuda()
        pairs.append((full[:, :n], p.b.cuda()))
        lams.append(p.lambdas.numpy())
        opts.append(tk.opts_default(sketch=tk.TK_SKETCH_GAUSS, s=max(2, n // 3) if low else min(4 * n, m), seed=k + 1,
                                    precond=tk.TK_PRECOND_LOWRANK if low else tk.TK_PRECOND_CHOL,
                                    precision=tk.TK_PREC_MIXED))
    Xs, infos, st = tk.tk_solve_batched(pairs, np.stack(lams), opts)
    assert st == tk.TK_OK
    for (A, b), lam, o, X, info in zip(pairs, lams, opts, Xs, infos):
        r = tk.tk_solve(A, b, lam, o)
        for i in range(N):
            e = float((X[i] - r.X[i]).norm() / r.X[i].norm())
            assert e < 2e-10, (tuple(A.shape), lam[i], e)  # each within 1e-10 of the minimiser
