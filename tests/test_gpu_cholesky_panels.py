"""The Cholesky trailing updates on the tensor cores: panels of 256 rows and the block rows inside them."""
import pytest
import torch

from paper_2203_07329_gb300 import tikhonov as tk

pytestmark = pytest.mark.gpu


# Orders with one panel, with a last panel of one, two, three and four block rows, ragged in the last 64, and
# several panels; columns in very different units.  R^T R differs from C + lambda I in entry (i, j) by at most
# n + 1 rounding errors of |R|^T |R| <= sqrt(c_ii c_jj); the check's own product adds n more, and a factor 2 for
# the digits' (8 2^-56) share.
@pytest.mark.parametrize("n,N", [(256, 2), (257, 1), (320, 3), (449, 2), (512, 2), (577, 5), (700, 1), (1100, 3),
                                 (2100, 2)])
def test_panel_updates_have_float64_backward_error(n, N):
    gen = torch.Generator().manual_seed(n)
    Y = torch.randn(2 * n, n, dtype=torch.float64, generator=gen).cuda()
    Y *= torch.pow(10.0, -6 * torch.rand(n, dtype=torch.float64, generator=gen)).cuda()
    C = Y.T @ Y
    lams = [10.0 ** -(3 * i + 12) for i in range(N)]
    R, brk = tk.tk_cholesky_shifted(C, lams, emulate=True)
    assert brk == [0] * N
    for i, lam in enumerate(lams):
        want = C + lam * torch.eye(n, dtype=torch.float64, device="cuda")
        d = want.diagonal().sqrt()
        err = ((R[i].T @ R[i] - want).abs() / (d[:, None] * d[None, :])).max().item()
        assert err < 4 * (n + 1) * 2.0 ** -53, err
        assert torch.tril(R[i], -1).abs().max().item() == 0.0


# More lambdas than the planes of one pass hold (2 GiB: 1638 of order 320): the factors on both sides of the
# border, same bound; and their inverses, which precondition neighbouring lambdas alike (iterations within 2).
def test_more_lambdas_than_one_pass():
    n, N, m = 270, 1650, 600
    gen = torch.Generator().manual_seed(1)
    A = torch.randn(m, n, dtype=torch.float64, generator=gen).cuda()
    b = torch.randn(m, dtype=torch.float64, generator=gen).cuda()
    C = A.T @ A
    lams = torch.logspace(-3, 1, N, dtype=torch.float64).numpy()
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    R, brk = tk.tk_cholesky_shifted(C, lams, emulate=True)
    assert brk == [0] * N
    for i in (0, 1637, 1638, N - 1):
        want = C + lams[i] * eye
        d = want.diagonal().sqrt()
        err = ((R[i].T @ R[i] - want).abs() / (d[:, None] * d[None, :])).max().item()
        assert err < 4 * (n + 1) * 2.0 ** -53, (i, err)
    r = tk.tk_solve(A, b, lams, tk.opts_default(precision=tk.TK_PREC_MIXED, sketch=tk.TK_SKETCH_GAUSS, s=m,
                                                max_refine=1))
    assert abs(r.info[1637]["iters"] - r.info[1638]["iters"]) <= 2
