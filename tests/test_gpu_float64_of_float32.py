"""The float64 form on float32 data, every sketch and both orientations, from the digit planes of A and without:
the solution of the widened data."""
import numpy as np
import pytest
import torch

from paper_2203_07329_gb300 import tikhonov as tk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sketch", [tk.TK_SKETCH_SRHT, tk.TK_SKETCH_GAUSS, tk.TK_SKETCH_SPARSE, tk.TK_SKETCH_SRDCT])
@pytest.mark.parametrize("m,n,pad", [(900, 31, 0), (5001, 130, 3), (40, 700, 1), (130, 5001, 0)])
def test_solves_as_the_widened_data(m, n, pad, sketch):
    gen = torch.Generator().manual_seed(m)
    full = torch.full((m, n + pad), float("nan"), dtype=torch.float32)
    full[:, :n] = torch.randn(m, n, generator=gen) / max(m, n) ** 0.5
    A = full.cuda()[:, :n]
    b = torch.randn(m, generator=gen, dtype=torch.float64).cuda()
    lams = np.geomspace(1e-3, 1.0, 3)
    o = tk.opts_default(sketch=sketch, s=6 * min(m, n))
    r = tk.tk_solve(A, b, lams, o)
    w = tk.tk_solve(A.double(), b, lams, o)
    assert r.status == tk.TK_OK and w.status == tk.TK_OK
    for i in range(3):  # both to the float64 accuracy of a problem of condition below 1e2
        assert float((r.X[i] - w.X[i]).norm()) <= 1e-12 * float(w.X[i].norm())
