"""tk_sketch_apply's float64 Gaussian sketch over the sizes at which a float64 solve forms its own from digit
planes of A (2^16 elements and more): it keeps the float64 pipe and agrees with the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from paper_2203_07329_gb300 import tikhonov as tk

pytestmark = pytest.mark.gpu


# just below, at and above 2^16 elements, above 2^19 (where the LSQR products use the planes too), both orientations
@pytest.mark.parametrize("m,n,s", [(1023, 64, 70), (1024, 64, 70), (4099, 33, 64), (9001, 61, 120), (64, 1024, 70),
                                   (61, 9001, 120)])
def test_gauss_sketch_matches_oracle(m, n, s):
    A = torch.randn(m, n, dtype=torch.float64, generator=torch.Generator().manual_seed(m + n))
    o = tk.opts_default(sketch=tk.TK_SKETCH_GAUSS, s=s, seed=8)
    Y = tk.tk_sketch_apply(A.cuda(), o).cpu().numpy()
    Yo = oracle.gauss_over(A.numpy(), 8, s) if m >= n else oracle.gauss_under(A.numpy(), 8, s)
    # entries agree to libm-vs-CUDA rounding (about 1e-16); sums differ in order
    np.testing.assert_allclose(Y, Yo, rtol=1e-12, atol=1e-12 * np.abs(Yo).max())
