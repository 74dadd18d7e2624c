"""tk_launch_count counts kernels: the replayed LSQR steps as many as the same steps launched one by one (which is how
they run under the profiler)."""
import pytest
import torch

from paper_2203_07329_gb300 import tikhonov as tk

pytestmark = pytest.mark.gpu


# one lambda (its slot count is the same either way); 9000 rows: the digits of a long vector start with a memset
@pytest.mark.parametrize("m,n,kw", [(9000, 70, {}), (900, 70, {}), (9000, 70, dict(precision=tk.TK_PREC_MIXED))])
def test_replays_count_kernels(m, n, kw):
    gen = torch.Generator().manual_seed(2)
    A = (torch.randn(m, n, generator=gen, dtype=torch.float64) / m ** 0.5).cuda()
    b = torch.randn(m, generator=gen, dtype=torch.float64).cuda()
    o = tk.opts_default(s=4 * n, **kw)

    def launches():
        c0 = tk.tk_launch_count()
        tk.tk_solve(A, b, [1e-2], o)
        return tk.tk_launch_count() - c0

    replayed = launches()
    tk.tk_profile_collect()
    tk.tk_profile_enable(True)
    try:
        direct = launches()
        tk.tk_profile_collect()
    finally:
        tk.tk_profile_enable(False)
    assert replayed == direct
