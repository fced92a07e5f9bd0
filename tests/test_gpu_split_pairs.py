"""The split GEMM's CTA-pair kernel at the edges of its tiles, chunks and K slices against the FP64
oracle.  Bounds: two FP16 parts leave at most 2^-23 of an element's leading power of two and
drop products below 2^-22, so with a few truncations per chunk and two levels of FP32 sums the
normwise error of normal operands stays below 6e-7; rows far below the operand's largest
element keep it relative to themselves down to 2^-16 (FP16's exponent range below 2^14)."""
import numpy as np
import pytest

import oracle
import synth
from helpers import empty_like_labels, from_dev, normwise, to_dev

pytestmark = pytest.mark.gpu

E = "C[m,n] = A[k,m] * B[k,n]"


@pytest.fixture(scope="module")
def comet():
    import paper_2102_06827_gb300 as c
    return c


def run(comet, expr, ext, arrays, **kw):
    import torch
    p = comet.Plan(expr, ext, torch.float32, precision="split_bf16", **kw)
    out = empty_like_labels([ext["m"], ext["n"]], torch.float32)
    p.contract([to_dev(a, np.float32) for a in arrays], out, p.workspace())
    comet.sync_status()
    return from_dev(out).astype(np.float64)


def f32(shape, seed, t, **kw):
    return synth.tensor(shape, seed, t, **kw).astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("ksplit", [1, 2])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (129, 49, 31), (257, 193, 65), (256, 192, 64), (255, 47, 129),
                                   (513, 385, 200), (300, 200, 4096), (300, 200, 4097)])
def test_tiles_chunks_and_slices(comet, M, N, K, ksplit):
    ext = dict(m=M, n=N, k=K)
    A, B = f32((K, M), 71, 0, kind="normal"), f32((K, N), 71, 1, kind="normal")
    assert normwise(run(comet, E, ext, [A, B], ksplit=ksplit), oracle.einsum(E, A, B)) <= 6e-7
    A, B = f32((K, M), 72, 0, kind="int", lo=-9, hi=9), f32((K, N), 72, 1, kind="int", lo=-9, hi=9)
    assert np.array_equal(run(comet, E, ext, [A, B], ksplit=ksplit), oracle.einsum(E, A, B))


def test_small_rows_keep_their_relative_precision(comet):
    ext = dict(m=200, n=96, k=300)
    A, B = f32((300, 200), 73, 0, kind="normal"), f32((300, 96), 73, 1, kind="normal")
    A = A * 2.0 ** -(np.arange(200) % 17)       # rows from the largest element's size to 2^-16 of it
    C, ref = run(comet, E, ext, [A, B]), oracle.einsum(E, A, B)
    rows = np.abs(C - ref).max(axis=1) / np.abs(ref).max(axis=1)
    assert rows.max() <= 1e-6


@pytest.mark.parametrize("views", [False, True])
@pytest.mark.parametrize("M,N,K", [(70, 50, 40), (700, 600, 300)])
def test_scale_slots_ignore_non_finite_elements(comet, M, N, K, views):
    # one block of the abs-max pass and many; an infinity and a NaN spoil their own rows only: the
    # operand's scale comes from its finite elements
    ext = dict(m=M, n=N, k=K)
    A, B = f32((K, M), 74, 0, kind="normal"), f32((K, N), 74, 1, kind="normal")
    A[:, 5] *= 2.0 ** 20
    ref = oracle.einsum(E, A, B)
    A[K // 2, 3], A[K - 1, M - 1] = np.inf, np.nan
    kw = {}
    if views:   # A inside a larger stored tensor of much larger values
        S = np.full((K + 3, M + 2), 1e30, order="F")
        S[2:K + 2, 1:M + 1] = A
        A, kw = S, dict(views=[(0, 0, K + 3, 2, 1), (0, 1, M + 2, 1, 1)])
    C = run(comet, E, ext, [A, B], ksplit=1, **kw)
    fine = np.ones(M, bool)
    fine[[3, M - 1]] = False
    assert normwise(C[fine], ref[fine]) <= 6e-7
    assert not np.isfinite(C[~fine]).any()


@pytest.mark.parametrize("expr", [E, "C[n,m] = A[k,m] * B[k,n]"])
@pytest.mark.parametrize("M,N,K", [(128 * 400 + 1, 48, 48), (128 * 400 + 1, 47, 96), (128 * 400 - 1, 48, 97),
                                   (128 * 400, 33, 128), (100, 3001, 96), (257, 191, 1000)])
def test_narrow_tiles_and_either_direction_of_the_result(comet, expr, M, N, K):
    # one group per tile up to 96 values of K and three groups above, rows of the result along M and along
    # N (odd extents: unaligned runs), stored and accumulated
    ext = dict(m=M, n=N, k=K)
    lhs = [M, N] if expr is E else [N, M]
    A, B = f32((K, M), 75, 0, kind="normal"), f32((K, N), 75, 1, kind="normal")
    ref = oracle.einsum(expr, A, B)
    import torch
    for scale in ("", "1.5 * ", "+"):
        e = expr.replace("= ", "+= 0.5 * ") if scale == "+" else expr.replace("= ", "= " + scale)
        p = comet.Plan(e, ext, torch.float32, precision="split_bf16", ksplit=1)
        C0 = f32(lhs, 75, 2, kind="normal")
        out = to_dev(C0, np.float32)
        p.contract([to_dev(a, np.float32) for a in (A, B)], out, p.workspace())
        comet.sync_status()
        want = C0 + 0.5 * ref if scale == "+" else (1.5 if scale else 1.0) * ref
        assert normwise(from_dev(out).astype(np.float64), want) <= 6e-7
