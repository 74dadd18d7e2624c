"""The float64 form's Gaussian sketch from digits where the embedding is taken in several blocks of columns: the same
sketch as on the float64 pipe, seen through the solutions and the iteration counts it gives."""
import pytest

from paper_2203_07329_gb300 import datagen, tikhonov as tk

pytestmark = pytest.mark.gpu


# two blocks with a ragged second one, m > n and m < n; three blocks of a result with too few tiles for the GPU (sums
# split along the block, too); one block and a second of a few columns
@pytest.mark.parametrize("m,n,s", [(32845, 600, 4096), (600, 32845, 4096), (80003, 40, 2500), (40, 80003, 2500),
                                   (21825, 70, 4096)])
def test_blocks_of_the_embedding(m, n, s):
    k, N = min(m, n), 2
    p = datagen.make_ridge_problem(m, n, datagen.spectrum("log", k, hi=1.0, lo=1e-3),
                                   datagen.log_lambdas(N, 1e-6, 1e-1), seed=m + n)
    A, b, lams = p.A.cuda(), p.b.cuda(), p.lambdas.numpy()
    assert max(m, n) > (1 << 31) // (24 * s) // 256 * 256  # beyond one block of 2 GiB, in whole chunks of 256 columns
    r1 = tk.tk_solve(A, b, lams, tk.opts_default(sketch=tk.TK_SKETCH_GAUSS, s=s))
    r0 = tk.tk_solve(A, b, lams, tk.opts_default(sketch=tk.TK_SKETCH_GAUSS, s=s, emulate_fp64=0))
    for i in range(N):
        assert r1.info[i]["status"] == 0 and r0.info[i]["status"] == 0
        assert float((r1.X[i] - r0.X[i]).norm()) <= 1e-10 * float(r0.X[i].norm())
        assert abs(r1.info[i]["iters"] - r0.info[i]["iters"]) <= 2
