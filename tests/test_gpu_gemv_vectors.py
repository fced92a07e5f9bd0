"""Tensor-times-vector steps at the edges of their 16-byte loads and of their K chunks (128 to 1024
values, by the size of the grid) against the FP64 oracle.  Bound: chunk sums carry twice FP32's
precision, so the result carries its final rounding and a second-order term: 2^-22 of sum |v x|."""
import numpy as np
import pytest

import oracle
import synth
from helpers import maxabs
from test_gpu_contract import run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def comet():
    import paper_2102_06827_gb300 as c
    return c


@pytest.mark.parametrize("expr", ["y[n] = A[n,k] * x[k]", "y[n] = A[k,n] * x[k]", "y[n] = A[n,l,k] * x[k,l]",
                                  "y[n] = A[k,n,l] * x[k,l]", "y[n] = A[n,k]"])
@pytest.mark.parametrize("N,K", [(4, 4), (4, 128), (132, 132), (128, 1028), (60, 3000), (1, 4096), (127, 129),
                                 (128, 126), (130, 128), (20000, 36), (9000, 1156)])
def test_vector_and_chunk_edges(comet, expr, N, K):
    ext = dict(n=N, k=K, l=3)
    labels = [t[t.index("[") + 1:t.index("]")].split(",") for t in expr.split("= ")[1].split(" * ")]
    ops = [synth.tensor([ext[l] for l in ls], 91, t, kind="normal").astype(np.float32)
           for t, ls in enumerate(labels)]
    C, _ = run(comet, expr, ext, ops, np.float32, precision="split_bf16")
    wide = [a.astype(np.float64) for a in ops]
    scale = float(np.max(oracle.abs_einsum(expr, *wide)))
    assert maxabs(C, oracle.einsum(expr, *wide)) <= 2.0 ** -22 * scale


@pytest.mark.parametrize("expr", ["y[n] = 0.0009765625 * A[n,k] * x[k]", "y[n] = 0.0009765625 * A[k,n] * x[k]"])
def test_chunk_sums_beyond_fp32(comet, expr):
    # sums of 1e40 that alpha brings back into range
    ext = dict(n=8, k=1024)
    A, x = np.full((8, 1024) if "n,k" in expr else (1024, 8), 1e37, np.float32), np.ones(1024, np.float32)
    C, _ = run(comet, expr, ext, [A, x], np.float32, precision="split_bf16")
    assert np.allclose(C, np.float64(np.float32(1e37)), rtol=2.0 ** -22)
