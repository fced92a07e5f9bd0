"""K slices of the emulated-FP64 GEMM: tiles beyond whole rounds over the SMs run in slices of whole
192-value chunks whose int64 sums a second kernel adds.  The sums are integers, so results on integer
operands are exact: fewer tiles than SMs, a few tiles past one round, more than half a round, last chunks
of 1 and 191 values, ragged tile edges, alpha and +=."""
import numpy as np
import pytest

import oracle
import synth
from helpers import from_dev, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(1, 1, 193), (130, 90, 1153), (257, 161, 767), (1400, 1200, 400),
                                   (1290, 1130, 385), (2100, 1010, 577)])
def test_integers_exact(M, N, K):
    import torch
    import paper_2102_06827_gb300 as comet
    e, ext = "C[m,n] += 0.5 * A[k,m] * B[n,k]", dict(m=M, n=N, k=K)
    A = synth.tensor((K, M), 91, 0, kind="int", lo=-2000, hi=2000)
    B = synth.tensor((N, K), 91, 1, kind="int", lo=-2000, hi=2000)
    C0 = synth.tensor((M, N), 91, 2, kind="int", lo=-9, hi=9)
    p = comet.Plan(e, ext, torch.float64, precision="emu_f64")
    out = to_dev(C0)
    p.contract([to_dev(A), to_dev(B)], out, p.workspace())
    comet.sync_status()
    assert np.array_equal(from_dev(out), C0 + 0.5 * oracle.einsum("C[m,n] = A[k,m] * B[n,k]", A, B))
