"""The x' scratch of original-space products grows with the number of columns: what it outgrows stays with
the handle, and a product's bits do not depend on the products before it."""
import pytest
import torch

from paper_2308_00106_gb300 import maxe
from paper_2308_00106_gb300 import workloads as W
from tests.test_gpu_order_scratch import CountingAllocator, _handle

pytestmark = pytest.mark.gpu

N = 5003


def _x(h, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(k)
    return torch.rand(h.cols, k, generator=g, device="cuda", dtype=h.vec_dtype) - 0.5


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_growth_frees_nothing_and_changes_no_bits(dtype):
    al = CountingAllocator()
    h, _, _ = _handle(N, dtype, al)
    made, freed = len(al.allocs), len(al.frees)
    ks = list(range(1, 65))
    first = {k: maxe.maxe_spmm(h, _x(h, k)) for k in ks}
    vb = 8 if dtype == "f64" else 4
    assert [b // (N * vb) for b in al.allocs[made:]] == [8, 16, 32, 64]
    assert len(al.frees) == freed
    for k in reversed(ks):  # now on the largest scratch
        assert torch.equal(maxe.maxe_spmm(h, _x(h, k)), first[k]), k
    h.close()
    assert not al.live


def test_growth_takes_less_where_memory_is_short():
    al = CountingAllocator()
    h, _, _ = _handle(N, "f32", al)
    maxe.maxe_spmm(h, _x(h, 16))
    want = maxe.maxe_spmm(h, _x(h, 17))
    h.close()
    al = CountingAllocator()
    h, _, _ = _handle(N, "f32", al)
    maxe.maxe_spmm(h, _x(h, 16))
    al.refuse = len(al.allocs)  # twice the sixteen columns
    assert torch.equal(maxe.maxe_spmm(h, _x(h, 17)), want)
    assert [b // (4 * N) for b in al.allocs[-2:]] == [32, 20]
    h.close()
    assert not al.live


def test_a_graph_survives_wider_products():
    A = W.poisson_uniform(7, N, 6.0, "f32", "cuda")
    h = maxe.from_csr(A, maxe.maxe_build_permutation(7, N, 0), maxe.maxe_build_permutation(7, N, 1))
    X, Y = _x(h, 8), torch.zeros(N, 8, device="cuda")
    first = maxe.maxe_spmm(h, X)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        maxe.maxe_spmm(h, X, Y)
    maxe.maxe_spmm(h, _x(h, 64))
    others = [torch.full((N, 8), 3.0, device="cuda") for _ in range(32)]  # would take any freed block
    graph.replay()
    assert torch.equal(Y, first)
    assert all(bool((t == 3.0).all()) for t in others)
    h.close()
