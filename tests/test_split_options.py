"""Options of the split GEMM's plan (host side): the accumulation-chunk limit, any number of K slices, and
the one-launch kernel's size limit."""
import time

import pytest

import paper_2102_06827_gb300 as comet

E = "C[m,n] = A[k,m] * B[k,n]"


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2102_06827_gb300 import build
    build.build()


def step(m, n, k, **kw):
    return comet.Plan(E, dict(m=m, n=n, k=k), "f32", precision="split_bf16", **kw).info["steps"][0]


@pytest.mark.parametrize("form", [-1, 0, 1])
@pytest.mark.parametrize("m,n,k", [(8, 1048560, 8), (8, 1048561, 8), (2, 2000000, 2), (2000000, 2, 2)])
def test_one_launch_kernel_only_where_its_grid_takes_the_size(m, n, k, form):
    st = step(m, n, k, form=form)
    long_n = (n if st["N"] == ["n"] else m) > 16 * 65535
    assert not (st["small"] and long_n)


@pytest.mark.parametrize("kc,chunk", [(0, 64), (1, 32), (32, 32), (63, 32), (64, 64), (1024, 64)])
def test_chunk_limit(kc, chunk):
    # long sums take chunks of 64 unless the caller asks for shorter ones
    assert step(512, 512, 6000, kc=kc, ksplit=1)["chunk"] == chunk
    assert step(512, 512, 4096, kc=kc, ksplit=1)["chunk"] == 32


@pytest.mark.parametrize("ksplit", [1000, 2 ** 31 - 1])
def test_any_number_of_k_slices_is_planned_at_once(ksplit):
    # more slices than K has stages, and partial sums that do not fit: the most that fit, without counting down
    t = time.perf_counter()
    st = step(1 << 14, 1 << 14, 4096, ksplit=ksplit)
    assert time.perf_counter() - t < 5.0
    assert 1 <= st["ksplit"] <= 64
    assert st["ksplit"] == step(1 << 14, 1 << 14, 4096, ksplit=64)["ksplit"]
