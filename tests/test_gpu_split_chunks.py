"""The caller's limit of the split GEMM's accumulation chunks reaches the kernel: shorter chunks give other
roundings of a long sum, inside the same bound (6e-7 normwise, as for the kernel's other sizes)."""
import numpy as np
import pytest

from helpers import empty_like_labels, from_dev, normwise, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,ksplit", [(300, 200, 4100, 1), (129, 49, 4800, 1), (256, 192, 12288, 2)])
def test_chunk_limit_reaches_the_kernel(M, N, K, ksplit):
    import torch
    import paper_2102_06827_gb300 as comet
    rng = np.random.default_rng(K)
    A, B = rng.uniform(0, 1, (K, M)).astype(np.float32), rng.uniform(0, 1, (K, N)).astype(np.float32)
    ref = A.astype(np.float64).T @ B.astype(np.float64)
    got = {}
    for kc in (0, 32, 64):
        p = comet.Plan("C[m,n] = A[k,m] * B[k,n]", dict(m=M, n=N, k=K), torch.float32, precision="split_bf16",
                       ksplit=ksplit, kc=kc)
        out = empty_like_labels([M, N], torch.float32)
        p.contract([to_dev(A), to_dev(B)], out, p.workspace())
        comet.sync_status()
        got[kc] = from_dev(out)
        assert normwise(got[kc], ref) <= 6e-7
    assert np.array_equal(got[0], got[64])
    assert not np.array_equal(got[0], got[32])
