"""Host-only checks (no GPU): the workspace queries of calls whose workspace the digit planes dominate stay within
what the header states for them, so that what fits the GPU as float64 data fits it as a solve."""
import ctypes as C

import pytest

GIB = float(1 << 30)


@pytest.fixture(scope="module")
def tk():
    from paper_2203_07329_gb300 import build
    build.build()
    from paper_2203_07329_gb300 import tikhonov
    tikhonov.lib()
    return tikhonov


def _prob(tk, m, n, dtype=None):
    # fake non-null device addresses: the queries do not touch them
    return tk.tk_problem(m, n, n, tk.TK_F64 if dtype is None else dtype, 0x1000, 0x2000)


def _size(tk, m, n, N, dtype=None, **kw):
    return tk.workspace_size(_prob(tk, m, n, dtype), N, tk.opts_default(**kw))


# tk_sketch_apply forms the float64 Gaussian sketch on the float64 pipe at every size: it has no digit planes of A
# to read, and its scratch is the embedding (8 s L bytes) and split planes of the small result
@pytest.mark.parametrize("m,n,s", [(1 << 17, 64, 256), (64, 1 << 17, 256)])
def test_sketch_apply_has_no_digit_planes(tk, m, n, s):
    out = C.c_size_t(0)
    o = tk.opts_default(sketch=tk.TK_SKETCH_GAUSS, s=s)
    assert tk.lib().tk_sketch_apply_workspace(C.byref(_prob(tk, m, n)), C.byref(o), C.byref(out)) == tk.TK_OK
    L = max(m, n)
    assert out.value <= 8 * s * L + 8 * m * n + (64 << 20)


# the float64 form widens float32 data first: the solve needs everything the same solve of float64 data needs
# (its sketch's and its transpose's buffers hold float64) and the widened copy
@pytest.mark.parametrize("sketch", [0, 1, 2, 3])
@pytest.mark.parametrize("m,n", [(65536, 1024), (4096, 60), (300, 1), (300, 20000), (20, 500)])
def test_float64_form_of_float32_data(tk, m, n, sketch):
    kw = dict(sketch=sketch, s=4 * min(m, n))
    assert _size(tk, m, n, 3, tk.TK_F32, **kw) >= _size(tk, m, n, 3, **kw) + 8 * m * n


# the SVD of the sketch from as many rows as any: no more than Y itself and the orthogonal start (two s x s matrices),
# which needs a row of s values in shared memory and is left out where none fits (s > 25600)
@pytest.mark.parametrize("s,n", [(25600, 25600), (25601, 25601), (60000, 60001)])
def test_svd_of_many_rows(tk, s, n):
    w = tk.lib().tk_sketch_svd_workspace(s, n)
    most = 8 * s * n + (16 * s * s if s <= 25600 else 0)
    assert 8 * s * n < w <= most + 8 * 32 * s + (1 << 20)


# the float64 form's Gaussian sketch from digits holds a bounded block of the embedding and its planes at a time: not
# 24 bytes for each of its s L values (2^20 x 2048: 192 GiB)
@pytest.mark.parametrize("m,n,s", [(1 << 20, 2048, 8192), (1 << 21, 2048, 8192), (2048, 1 << 20, 8192),
                                   (1 << 20, 64, 60000)])
def test_gaussian_sketch_of_the_float64_form(tk, m, n, s):
    srht = _size(tk, m, n, 4, sketch=tk.TK_SKETCH_SRHT, s=s)
    assert _size(tk, m, n, 4, sketch=tk.TK_SKETCH_GAUSS, s=s) <= srht + 4 * GIB


# the LSQR vectors of very many lambdas get no digit planes beyond 64 GiB: the solve takes what it takes without digits
def test_no_vector_planes_beyond_64_gib(tk):
    o = dict(s=256)
    assert _size(tk, 1 << 20, 64, 4097, **o) <= _size(tk, 1 << 20, 64, 4097, emulate_fp64=0, **o) + GIB
    assert _size(tk, 1 << 20, 64, 4096, **o) >= _size(tk, 1 << 20, 64, 4096, emulate_fp64=0, **o) + 64 * GIB


def _batched(tk, m, n, N, P, **kw):
    ps = (tk.tk_problem * P)(*[_prob(tk, m, n) for _ in range(P)])
    o, out = tk.opts_default(**kw), C.c_size_t(0)
    assert tk.lib().tk_workspace_size_batched(C.byref(ps), P, N, C.byref(o), 1, C.byref(out)) == tk.TK_OK
    return out.value


# float64 problems on the host lanes: the digit planes of all lanes together stay within 32 GiB (or one problem's), so
# that 8 problems of 8 GiB each still fit the GPU beside their workspace; small ones keep 8 lanes
def test_lanes_of_large_float64_problems(tk):
    m, n, N = 1 << 19, 2048, 4
    for sketch in (tk.TK_SKETCH_SRHT, tk.TK_SKETCH_GAUSS):
        o = dict(sketch=sketch, s=8192)
        assert _batched(tk, m, n, N, 8, **o) + 8 * 8 * m * n <= 200 * GIB
        assert _batched(tk, m, n, N, 8, **o) == 2 * _batched(tk, m, n, N, 1, **o)
    one = _batched(tk, 4096, 256, N, 1, s=1024)
    assert _batched(tk, 4096, 256, N, 8, s=1024) == 8 * one
    one = _batched(tk, 1 << 17, 2048, N, 1, s=8192)  # 2^28 elements
    assert _batched(tk, 1 << 17, 2048, N, 8, s=8192) == 8 * one
    one = _batched(tk, m, n, N, 1, s=8192, emulate_fp64=0)
    assert _batched(tk, m, n, N, 8, s=8192, emulate_fp64=0) == 8 * one
