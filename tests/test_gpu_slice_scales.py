"""K slices of the split GEMM at operand scales and alphas far from one: the slices' partial sums are FP32
words, the result's scale is not in them.

Bound: the split precision's 1e-6 normwise against FP64."""
import numpy as np
import pytest

from helpers import empty_like_labels, from_dev, normwise, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,M,N,K,ksplit,ea,eb,alpha", [
    (np.float64, 256, 256, 480, 0, -100, -110, 1.0),    # planner's own slices
    (np.float64, 256, 256, 480, 0, 300, -200, 1.0),
    (np.float64, 130, 50, 200, 2, 100, 90, -2.0),
    (np.float64, 130, 50, 200, 2, -500, -400, 2.0 ** 300),
    (np.float32, 130, 50, 200, 2, -80, -90, 2.0 ** 120),
    (np.float32, 130, 50, 200, 3, 70, 80, 2.0 ** -100),
    (np.float32, 256, 256, 1024, 0, -3, 5, 1.0),
])
def test_scale_is_applied_after_the_slices_are_added(dtype, M, N, K, ksplit, ea, eb, alpha):
    import torch
    import paper_2102_06827_gb300 as comet
    rng = np.random.default_rng(K)
    A = np.ldexp(rng.uniform(-1, 1, (K, M)), ea).astype(dtype).astype(np.float64)
    B = np.ldexp(rng.uniform(-1, 1, (K, N)), eb).astype(dtype).astype(np.float64)
    tdt = torch.float32 if dtype == np.float32 else torch.float64
    p = comet.Plan("C[m,n] = A[k,m] * B[k,n]", dict(m=M, n=N, k=K), tdt, precision="split_bf16", ksplit=ksplit,
                   alpha=alpha)
    st = p.info["steps"][0]
    assert st["ksplit"] > 1 and not st["small"]
    out = empty_like_labels([M, N], tdt)
    p.contract([to_dev(A, dtype), to_dev(B, dtype)], out, p.workspace())
    comet.sync_status()
    ref = alpha * (A.T @ B)
    assert normwise(from_dev(out), ref) <= 1e-6
