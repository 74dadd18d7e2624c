"""The float64 form's products with A from exact digits on the tensor cores (emulate_fp64 = 1): the
same solutions as on the float64 pipe (emulate_fp64 = 0), whatever the shape and the scales of A."""
import math

import numpy as np
import pytest
import torch

from paper_2203_07329_gb300 import datagen, tikhonov as tk

pytestmark = pytest.mark.gpu


def _solve(A, b, lams, **kw):
    return tk.tk_solve(A, b, lams, tk.opts_default(**kw))


# A at and around the smallest size that is split into digits (2^19 elements), ragged against the 64-,
# 128- and 256-value tiles, one and several tiles of 32 lambdas, float64 views with odd row strides,
# the explicit inverse over one to three doubling levels with ragged last blocks (257 .. 1100 columns), more
# row tiles than SMs (60001 rows: a CTA's rings and buffers run on over several tiles), and m < n with vectors
# of 1, 2, 4 and 8 CTAs per v-step.  Both forms solve to the float64 accuracy of the problem (condition about
# 1e3: 1e-10).
@pytest.mark.parametrize("m,n,N,pad", [(8192, 64, 2, 0), (8192, 65, 1, 0), (8193, 65, 3, 1), (2051, 257, 33, 0), (1500, 700, 5, 3),
                                       (16500, 40, 4, 0), (129, 4099, 4, 0), (500, 1100, 34, 5), (63, 8400, 2, 0),
                                       (101, 17001, 3, 0), (6000, 1100, 3, 0), (517, 4000, 2, 0),
                                       (60001, 130, 3, 0)])
def test_digit_solve_matches_float64_pipe(m, n, N, pad):
    k = min(m, n)
    p = datagen.make_ridge_problem(m, n, datagen.spectrum("log", k, hi=1.0, lo=1e-3),
                                   datagen.log_lambdas(N, 1e-6, 1e-1), seed=m + n)
    full = torch.full((m, n + pad), float("nan"), dtype=torch.float64, device="cuda")
    full[:, :n] = p.A.cuda()
    A, b, lams = full[:, :n], p.b.cuda(), p.lambdas.numpy()
    s = min(4 * k, max(m, n))
    r1 = _solve(A, b, lams, sketch=tk.TK_SKETCH_SRHT, s=s)
    r0 = _solve(A, b, lams, sketch=tk.TK_SKETCH_SRHT, s=s, emulate_fp64=0)
    for i in range(N):
        e = float((r1.X[i] - r0.X[i]).norm() / r0.X[i].norm())
        assert e < 1e-10, (lams[i], e)
        assert r1.info[i]["status"] == 0
        assert abs(r1.info[i]["iters"] - r0.info[i]["iters"]) <= 2


# rows and columns of A in very different units: the digits follow both, so every entry of the two
# products keeps the accuracy of a float64 sum of its own terms (K terms, each relative to the
# product of the scaled maxima: 8 2^-53 sqrt(K) of sum |a||x| as for the other digit products)
@pytest.mark.parametrize("rows,cols", [(0, 12), (12, 0), (9, 9)])
def test_digit_products_follow_row_and_column_scales(rows, cols):
    gen = torch.Generator().manual_seed(3)
    m, n, M = 3001, 390, 5
    A = torch.randn(m, n, generator=gen, dtype=torch.float64)
    A *= torch.pow(10.0, -rows * torch.rand(m, 1, generator=gen, dtype=torch.float64))
    A *= torch.pow(10.0, -cols * torch.rand(1, n, generator=gen, dtype=torch.float64))
    # x in the units of the columns, b in those of the rows, as the solution of a fit has them
    X = torch.randn(M, n, generator=gen, dtype=torch.float64) / A.abs().amax(0)
    b = torch.zeros(m, dtype=torch.float64)
    R, G = tk.tk_residual(A.cuda(), b.cuda(), X.cuda(), True, with_g=True)
    R, G, Ah, Xh = R.cpu().numpy(), G.cpu().numpy(), A.numpy(), X.numpy()
    Rref = -(Xh.astype(np.longdouble) @ Ah.T.astype(np.longdouble))
    err = np.max(np.abs((R - Rref).astype(np.float64)) / (np.abs(Xh) @ np.abs(Ah).T))
    assert err < 8 * 2.0 ** -53 * math.sqrt(n), err
    Gref = R.astype(np.longdouble) @ Ah.astype(np.longdouble)
    err = np.max(np.abs((G - Gref).astype(np.float64)) / (np.abs(R) @ np.abs(Ah)))
    assert err < 8 * 2.0 ** -53 * math.sqrt(m), err


# the same levels in float32 (the mixed form's preconditioner): refined to the float64 solution, with as
# many iterations as the float32 pipe's inverse gives
# (the last two: 20 and 40 lambdas over more row tiles than the GPU has slots for)
@pytest.mark.parametrize("n,N,m", [(256, 3, 1041), (300, 1, 1217), (513, 5, 2069), (1100, 3, 4417), (1290, 2, 5177),
                                   (100, 20, 80001), (100, 40, 80001)])
def test_mixed_digits(n, N, m):
    p = datagen.make_ridge_problem(m, n, datagen.spectrum("log", n, hi=1.0, lo=1e-4),
                                   datagen.log_lambdas(N, 1e-6, 1e-1), seed=n)
    A, b, lams = p.A.cuda(), p.b.cuda(), p.lambdas.numpy()
    kw = dict(sketch=tk.TK_SKETCH_GAUSS, s=3 * n, precision=tk.TK_PREC_MIXED)
    r1 = _solve(A, b, lams, **kw)
    r0 = _solve(A, b, lams, lsqr_tc=0, emulate_fp64=0, **kw)
    for i in range(N):
        e = float((r1.X[i] - r0.X[i]).norm() / r0.X[i].norm())
        assert e < 2e-10, (lams[i], e)  # each within 1e-10 of the minimiser
        assert r1.info[i]["iters"] <= 1.2 * r0.info[i]["iters"] + 3


def test_non_finite_a_is_enumeric_from_digits():
    gen = torch.Generator().manual_seed(5)
    A = torch.randn(9000, 70, generator=gen, dtype=torch.float64)
    b = torch.randn(9000, generator=gen, dtype=torch.float64).cuda()
    A[4001, 3] = float("nan")
    r = tk.tk_solve(A.cuda(), b, [1e-2, 1.0], tk.opts_default(sketch=tk.TK_SKETCH_SRHT, s=280),
                    allow=tuple(range(8)))
    assert r.status == tk.TK_ENUMERIC


# the low-rank preconditioner's apply over slot counts around its groups of 8 slots, ragged rows and columns, and
# more sketch rows than fit in shared memory with 8 slots (s > 2560): the same solutions as with the Cholesky one
@pytest.mark.parametrize("m,n,s,N", [(3000, 301, 97, 1), (5001, 333, 120, 9), (2500, 257, 64, 17), (6000, 2600, 2570, 3)])
def test_lowrank_apply_shapes(m, n, s, N):
    p = datagen.make_ridge_problem(m, n, datagen.spectrum("exp", n, tau=n / 40.0), datagen.log_lambdas(N, 1e-3, 1.0),
                                   seed=m)
    A, b, lams = p.A.cuda(), p.b.cuda(), p.lambdas.numpy()
    r1 = _solve(A, b, lams, sketch=tk.TK_SKETCH_GAUSS, s=s, precond=tk.TK_PRECOND_LOWRANK)
    r0 = _solve(A, b, lams, sketch=tk.TK_SKETCH_GAUSS, s=min(4 * n, m), emulate_fp64=0)
    for i in range(N):
        e = float((r1.X[i] - r0.X[i]).norm() / r0.X[i].norm())
        assert e < 1e-10, (lams[i], e)
        assert r1.info[i]["status"] == 0


# A spectrum down to 1e-8 and lambda down to 1e-10 (1e-12): the factors' diagonals span five (six) decades, and
# the explicit inverse must precondition as the one from the SIMT pipes does (equal iterations up to rounding)
@pytest.mark.parametrize("mixed,n,lo", [(True, 700, 1e-10), (True, 1500, 1e-10), (False, 1100, 1e-12)])
def test_digit_inverse_of_small_lambdas(mixed, n, lo):
    m, N = 6 * n, 6
    p = datagen.make_ridge_problem(m, n, datagen.spectrum("log", n, hi=1.0, lo=1e-8),
                                   datagen.log_lambdas(N, lo, 1e-2), seed=n)
    A, b, lams = p.A.cuda(), p.b.cuda(), p.lambdas.numpy()
    kw = dict(sketch=tk.TK_SKETCH_GAUSS, s=3 * n, precision=tk.TK_PREC_MIXED if mixed else tk.TK_PREC_FP64)
    r1 = _solve(A, b, lams, **kw)
    r0 = _solve(A, b, lams, lsqr_tc=0, emulate_fp64=0, **kw)
    for i in range(N):
        assert r1.info[i]["status"] == r0.info[i]["status"], lams[i]
        assert r1.info[i]["iters"] <= 1.2 * r0.info[i]["iters"] + 3, (lams[i], r1.info[i], r0.info[i])
