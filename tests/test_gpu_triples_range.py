"""The FP32 triples energy where FP32 sums of its terms do not reach: totals above FP32's range, an
infinite term, and terms whose leading parts cancel.  One term of the nine is non-zero and one operand is
constant, so T and the energies are known in closed form.

Bounds: T is exact; each T^2 / D and each thread's sum of 16 has at most 32 roundings of 2^-24 (the
division's two units included), everything beyond is exact to 2^-47."""
import numpy as np
import pytest

from triples_terms import LABELS, SIGNS, T_LABELS, operand_labels, terms

pytestmark = pytest.mark.gpu


def energy(ext, x, eps):
    """Energy of one block: the first term's X operand is x (its labels' extents), its Y all ones."""
    import torch
    import paper_2102_06827_gb300 as comet
    plan = comet.TriplesPlan(terms(), LABELS, [[ext[l] for l in LABELS]], SIGNS, torch.float32)
    assert plan.info["tensor_core"]
    keep = []
    for p, e in enumerate(terms()):
        for q, ls in enumerate(operand_labels(e)):
            shape = tuple(ext[l] for l in ls)
            v = np.zeros(shape) if p else np.ones(shape) if q else np.broadcast_to(x, shape)
            keep.append(torch.from_numpy(np.ravel(v, order="F").astype(np.float32)).cuda())
    keep_e = [torch.from_numpy(np.asarray(eps[l], dtype=np.float32)).cuda() for l in T_LABELS]
    en, ws = torch.empty(1, dtype=torch.float64, device="cuda"), plan.workspace()
    plan.prepare(ws)
    plan.energy(torch.tensor([t.data_ptr() for t in keep], dtype=torch.int64, device="cuda"),
                torch.tensor([t.data_ptr() for t in keep_e], dtype=torch.int64, device="cuda"), en, ws)
    comet.sync_status()
    return float(en.item())


def flat_eps(ext, virt, occ):
    return {l: np.full(ext[l], virt if l in "abc" else occ) for l in T_LABELS}


@pytest.mark.parametrize("sizes", [(8, 4, 4, 4, 4, 4), (13, 6, 5, 7, 4, 9)])
def test_total_above_fp32_range(sizes):
    ext = dict(zip(T_LABELS, sizes), d=1)
    e = energy(ext, 2.0 ** 62, flat_eps(ext, 1.0, -1.0))   # every term -2^124 / 6, a thread's sum below 6e37
    ref = -float(np.prod(sizes)) * 2.0 ** 124 / 6
    assert abs(ref) > 3.5e38
    assert abs(e - ref) <= 32 * 2.0 ** -24 * abs(ref)


def test_zero_denominator_gives_an_infinite_energy():
    ext = dict(a=3, b=2, c=2, i=2, j=2, k=2, d=1)
    eps = flat_eps(ext, 1.0, -1.0)
    for l in T_LABELS:
        eps[l][0] = 0.0            # D = 0 at the first element alone, elsewhere below zero
    assert np.isinf(energy(ext, 1.0, eps))


def test_leading_parts_that_cancel():
    # terms 1, -1 and 2^-30: what is left of the sum is in its rounding errors
    ext = dict(a=3, b=1, c=1, i=1, j=1, k=1, d=1)
    eps = flat_eps(ext, 0.0, 0.0)
    eps["a"] = np.array([-1.0, 1.0, -1.0])                 # D = 1, -1, 1
    x = np.array([1.0, 1.0, 2.0 ** -15])[None, :, None, None]   # [d, a, b, i]
    assert energy(ext, x, eps) == 2.0 ** -30
