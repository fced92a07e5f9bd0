"""Small contractions: the one-launch FP32 kernel of the split precision and the narrow FP64 tiles,
at their tile, K-chunk and K-tail edges against the FP64 oracle.

Bounds: the FP32 kernel keeps the rounding error of every addition, so the result carries the final
rounding and the errors' own (2^-24 of sums that are themselves 2^-24 of the result, plus one
uncompensated rounding while a product exceeds its running sum): 4 units of 2^-24 normwise.  FP64:
K additions of 2^-53."""
import numpy as np
import pytest

import oracle
import synth
from helpers import empty_like_labels, from_dev, normwise, to_dev

pytestmark = pytest.mark.gpu

EXPRS = ["C[m,n] = A[k,m] * B[k,n]", "C[m,n] = A[m,k] * B[n,k]", "C[n,m] = A[m,k] * B[k,n]"]
SIZES = [(1, 1, 1), (16, 16, 256), (17, 15, 257), (33, 47, 255), (5, 100, 513), (90, 70, 7), (576, 560, 23)]


@pytest.fixture(scope="module")
def comet():
    import paper_2102_06827_gb300 as c
    return c


def run(comet, expr, ext, arrays, dtype, precision, out_init=None):
    import torch
    p = comet.Plan(expr, ext, torch.float32 if dtype == np.float32 else torch.float64, precision=precision)
    labels = expr[expr.index("[") + 1:expr.index("]")].split(",")
    out = to_dev(out_init, dtype) if out_init is not None else empty_like_labels([ext[l] for l in labels],
                                                                                 p.dtype)
    p.contract([to_dev(a, dtype) for a in arrays], out, p.workspace())
    comet.sync_status()
    return from_dev(out).astype(np.float64), p


def shapes(expr, ext):
    _, _, _, _, ops = oracle.parse(expr)
    return [tuple(ext[l] for l in ls) for _, ls in ops]


@pytest.mark.parametrize("expr", EXPRS)
@pytest.mark.parametrize("M,N,K", SIZES)
def test_fp32_kernel(comet, expr, M, N, K):
    ext = dict(m=M, n=N, k=K)
    arrays = [synth.tensor(s, 81, t, kind="normal").astype(np.float32).astype(np.float64)
              for t, s in enumerate(shapes(expr, ext))]
    C, p = run(comet, expr, ext, arrays, np.float32, "split_bf16")
    if M * N * K < 1e6:
        assert p.info["steps"][0].get("small") or p.info["steps"][0]["kernel"] == "gemv"
    assert normwise(C, oracle.einsum(expr, *arrays)) <= 4 * 2.0 ** -24
    C0 = np.round(4 * synth.tensor(C.shape, 81, 9)).astype(np.float32).astype(np.float64)
    ints = [synth.tensor(s, 82, t, kind="int", lo=-5, hi=5) for t, s in enumerate(shapes(expr, ext))]
    C, _ = run(comet, expr.replace("= ", "-= 1.5 * "), ext, ints, np.float32, "split_bf16", out_init=C0)
    assert np.array_equal(C, C0 - 1.5 * oracle.einsum(expr, *ints))


def test_fp32_kernel_partial_sums_out_of_range(comet):
    # products of 1e40 that cancel exactly: the result is finite although FP32 products are not
    A = np.array([[1e20, -1e20, 3.0], [1.0, 2.0, -4.0]]).T   # [k, m]
    B = np.array([[1e20, 1e20, 2.0], [0.5, 0.25, 1.0]]).T
    C, _ = run(comet, EXPRS[0], dict(m=2, n=2, k=3), [A, B], np.float32, "split_bf16")
    ref = oracle.einsum(EXPRS[0], A.astype(np.float32).astype(np.float64), B.astype(np.float32).astype(np.float64))
    assert np.allclose(C, ref, rtol=1e-6)


@pytest.mark.parametrize("expr", EXPRS)
@pytest.mark.parametrize("M,N,K", SIZES)
def test_fp64_tiles(comet, expr, M, N, K):
    ext = dict(m=M, n=N, k=K)
    arrays = [synth.tensor(s, 83, t, kind="normal") for t, s in enumerate(shapes(expr, ext))]
    C, _ = run(comet, expr, ext, arrays, np.float64, "native")
    assert normwise(C, oracle.einsum(expr, *arrays)) <= max(4, K) * 2.0 ** -53
