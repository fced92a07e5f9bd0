"""The small FP32 contractions at the ends of FP32's range: products far below it that alpha brings back,
operands of subnormal and of very different magnitude, zero rows, and the sizes that one launch cannot
take.

Bounds.  In the normal range 4 units of 2^-24 normwise, as in the kernel's other tests (the rounding errors
of all additions are kept).  Each row and column of a tile has its own power of two, so the bound holds for
every row by itself.  A result below FP32's normal range has FP32's spacing there: half of 2^-149."""
import numpy as np
import pytest

import oracle
from helpers import empty_like_labels, from_dev, normwise, to_dev

pytestmark = pytest.mark.gpu

E = "C[m,n] = A[k,m] * B[k,n]"


def run(A, B, alpha=1.0, expr=E, **kw):
    import torch
    import paper_2102_06827_gb300 as comet
    ext = dict(k=A.shape[0], m=A.shape[1], n=B.shape[1])
    if expr != E:
        A, B = A.T, B.T
    p = comet.Plan(expr, ext, torch.float32, precision="split_bf16", alpha=alpha, **kw)
    out = empty_like_labels([ext["m"], ext["n"]], torch.float32)
    p.contract([to_dev(A, np.float32), to_dev(B, np.float32)], out, p.workspace())
    comet.sync_status()
    return from_dev(out).astype(np.float64), p.info["steps"][0]


def f32(x):
    return np.asarray(x, dtype=np.float32).astype(np.float64)


@pytest.mark.parametrize("expr", [E, "C[m,n] = A[m,k] * B[n,k]"])
@pytest.mark.parametrize("M,N,K", [(16, 16, 1), (17, 33, 257), (40, 24, 600)])
@pytest.mark.parametrize("ea,eb,alpha", [(-76, -76, 1e30), (-66, -66, 1e30), (-100, -120, 2.0 ** 100),
                                         (-140, -10, 1e25), (-60, -67, 1.0), (-80, 20, -3.0)])
def test_products_below_the_range(expr, M, N, K, ea, eb, alpha):
    rng = np.random.default_rng(M + K)
    A, B = f32(np.ldexp(rng.normal(size=(K, M)), ea)), f32(np.ldexp(rng.normal(size=(K, N)), eb))
    C, step = run(A, B, alpha, expr)
    assert step["small"]
    ref = alpha * (A.T @ B)
    assert np.all(np.isfinite(C))
    assert np.abs(C - ref).max() <= 4 * 2.0 ** -24 * np.abs(ref).max() + 2.0 ** -150


def test_rows_of_different_magnitude():
    # every second row of A and column of B is tiny, some are zero: the tiny ones' products meet alpha alone
    rng = np.random.default_rng(9)
    M, N, K = 50, 37, 300
    A, B = rng.normal(size=(K, M)), rng.normal(size=(K, N))
    A[:, ::2] = np.ldexp(A[:, ::2], -75)
    B[:, ::2] = np.ldexp(B[:, ::2], -75)
    A[:, 4] = 0.0
    B[:, 6] = 0.0
    A, B = f32(A), f32(B)
    C, step = run(A, B, 2.0 ** 60)
    assert step["small"]
    ref = 2.0 ** 60 * (A.T @ B)
    for i in (0, 1):
        for j in (0, 1):
            assert normwise(C[i::2, j::2], ref[i::2, j::2]) <= 4 * 2.0 ** -24, (i, j)
    assert np.all(C[4] == 0) and np.all(C[:, 6] == 0)


def test_infinite_element_beside_tiny_ones():
    A = np.full((3, 4), 1e-25)
    B = np.full((3, 5), 1e-25)
    A[1, 2] = np.inf
    C, _ = run(A, B, 1e30)
    ref = 1e30 * (f32(A).T @ f32(B))
    assert np.all(np.isinf(C[2])) and np.allclose(C[[0, 1, 3]], ref[[0, 1, 3]], rtol=1e-6, atol=0)


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("m,n,k", [(8, 1048560, 8), (8, 1048561, 8), (2, 1100000, 3)])
def test_long_dimension_in_either_form(m, n, k, form):
    # the one-launch kernel takes N up to 65535 tiles of 16; the forms put either dimension there
    rng = np.random.default_rng(n + form)
    A, B = f32(rng.normal(size=(k, m))), f32(rng.normal(size=(k, n)))
    C, step = run(A, B, form=form)
    assert normwise(C, A.T @ B) <= 6e-7
