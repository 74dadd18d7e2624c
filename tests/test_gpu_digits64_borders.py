"""The float64 form around the sizes at which its digit routes begin: 2^16 elements of A (planes for the Gaussian
sketch, digits for the Gram matrix, the factors' updates and their inverse) and 2^19 (the LSQR products, too)."""
import pytest
import torch

from paper_2203_07329_gb300 import datagen, tikhonov as tk

pytestmark = pytest.mark.gpu


# just below 2^16 elements, at it and above; just below 2^19, at it and above; odd sizes and padded row strides; both
# orientations; orders beyond 256 (levels of the inverse, panels) on both sides of 2^19.  Both forms solve to the
# float64 accuracy of the problem (condition about 1e3: 1e-10) with the same iteration counts.
@pytest.mark.parametrize("sketch", [tk.TK_SKETCH_GAUSS, tk.TK_SKETCH_SRHT])
@pytest.mark.parametrize("m,n,pad", [(1023, 64, 0), (1024, 64, 0), (1111, 59, 3), (8191, 64, 0), (8192, 64, 1),
                                     (1001, 260, 0), (1301, 403, 5), (4099, 33, 0), (64, 1023, 0), (64, 1024, 0),
                                     (59, 1111, 3), (64, 8191, 1), (64, 8192, 0), (301, 1201, 0), (403, 1301, 5)])
def test_borders_of_the_digit_routes(m, n, pad, sketch):
    k, N = min(m, n), 3
    p = datagen.make_ridge_problem(m, n, datagen.spectrum("log", k, hi=1.0, lo=1e-3),
                                   datagen.log_lambdas(N, 1e-6, 1e-1), seed=m + n)
    full = torch.full((m, n + pad), float("nan"), dtype=torch.float64, device="cuda")
    full[:, :n] = p.A.cuda()
    A, b, lams = full[:, :n], p.b.cuda(), p.lambdas.numpy()
    o = dict(sketch=sketch, s=min(4 * k, max(m, n)))
    r1 = tk.tk_solve(A, b, lams, tk.opts_default(**o))
    r0 = tk.tk_solve(A, b, lams, tk.opts_default(emulate_fp64=0, **o))
    for i in range(N):
        assert r1.info[i]["status"] == 0 and r0.info[i]["status"] == 0
        assert float((r1.X[i] - r0.X[i]).norm()) <= 1e-10 * float(r0.X[i].norm())
        assert abs(r1.info[i]["iters"] - r0.info[i]["iters"]) <= 2
