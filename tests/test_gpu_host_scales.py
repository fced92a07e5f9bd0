"""Scales of the host pipeline's slices: every slice of an operand has its own power of two, and the
GEMM blocks read those of both their slices, whatever lies next to them in the workspace.  The sizes
put the end of the workspace within the last 2.4 KB of the 32 MiB that the no-alloc entry has, where there is
no room for the abs-max slots but beside the scale words.

Bounds: those of the precisions (split 1e-6, emulated FP64 1e-12, normwise), here for each block by
itself, since a block's error is relative to the largest elements of its own two slices."""
import numpy as np
import pytest

from helpers import normwise

pytestmark = pytest.mark.gpu

LIMIT = 32 << 20


@pytest.mark.parametrize("m,n,k,precision", [
    (2730, 2731, 1024, "split_bf16"), (3413, 2048, 1024, "split_bf16"),
    (5461, 5461, 256, "emu_f64"), (2730, 8192, 256, "emu_f64"),
])
def test_every_block_has_its_own_slices_scales(m, n, k, precision):
    import torch
    import paper_2102_06827_gb300 as comet
    dtype = torch.float64 if precision == "emu_f64" else torch.float32
    p = comet.Plan("C[m,n] = A[k,m] * B[k,n]", dict(m=m, n=n, k=k), dtype, precision=precision)
    assert LIMIT - 2432 < p.workspace_bytes <= LIMIT
    hp = p.info["host_pipe"]
    assert hp["slices"] > 1
    bounds = {hp["label"]: hp["bounds"], hp["w_label"]: hp["w_bounds"]}
    rng = np.random.default_rng(5)
    ops = []
    for label, rows, first in (("m", m, -9), ("n", n, 3)):   # torch row-major: [rows][k], k fastest
        x = rng.uniform(-1, 1, (rows, k))
        for i, (lo, hi) in enumerate(zip(bounds[label], bounds[label][1:])):
            x[lo:hi] *= 2.0 ** (first + 5 * i)               # every slice in another binade
        ops.append(torch.from_numpy(x).to(dtype).pin_memory())
    out = torch.zeros((n, m), dtype=dtype).pin_memory()
    p.contract_host(ops, out, [torch.empty_like(t, device="cuda") for t in ops],
                    torch.empty((n, m), dtype=dtype, device="cuda"), p.workspace())
    ref = ops[1].double().numpy() @ ops[0].double().numpy().T
    got = out.numpy()
    tol = 1e-12 if precision == "emu_f64" else 1e-6
    for n0, n1 in zip(bounds["n"], bounds["n"][1:]):
        for m0, m1 in zip(bounds["m"], bounds["m"][1:]):
            assert normwise(got[n0:n1, m0:m1], ref[n0:n1, m0:m1]) <= tol, (m0, n0)
