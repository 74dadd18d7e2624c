"""Float64 problems whose digit planes allow fewer host lanes than there are problems: the solutions of single solves."""
import pytest
import torch

from paper_2203_07329_gb300 import tikhonov as tk

pytestmark = pytest.mark.gpu


def test_fewer_lanes_than_problems():
    m, n, P = (1 << 22) + 64, 64, 8  # just above 4 GiB of planes each: 7 lanes within 32 GiB
    gen = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randn(m, n, generator=gen, dtype=torch.float64, device="cuda")
    bs = [torch.randn(m, generator=gen, dtype=torch.float64, device="cuda") for _ in range(P)]
    o = tk.opts_default(sketch=tk.TK_SKETCH_SPARSE, s=1024)
    one = tk.workspace_size(tk.make_problem(A, bs[0]), 2, o)
    assert 7 * one <= tk.workspace_size_batched([(A, b) for b in bs], 2, o) < 7 * (one + 256) + 256
    lams = [[0.01 * (p + 1), 1.0] for p in range(P)]
    Xs, _, st = tk.tk_solve_batched([(A, b) for b in bs], lams, o)
    assert st == tk.TK_OK
    for p in range(P):
        r = tk.tk_solve(A, bs[p], lams[p], o)
        assert float((Xs[p] - r.X).norm()) <= 1e-10 * float(r.X.norm())
