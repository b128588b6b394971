"""Original-space products whose y rows are put in order by a second pass, against
the permuted product and a handle that scatters; replayed from a graph.  Rows
have at most 17 entries, |a| <= 1, |x| <= 1/2: two orders of a row's sum differ by
at most 2 * 18 * 2^-24 * 8.5 < 2e-5."""
import pytest
import torch

from paper_2308_00106_gb300 import maxe
from paper_2308_00106_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N = 1_900_001  # 16-byte rows: 30.4 MB of Y, just past the line


@pytest.fixture(scope="module")
def handles():
    A = W.poisson_uniform(3, N, 3.0, "f32", "cuda")
    r, c = maxe.maxe_build_permutation(1, N, 0), maxe.maxe_build_permutation(1, N, 1)
    tuned = maxe.from_csr(A, r, c, autotune=True)
    yield tuned, r, c
    tuned.close()


@pytest.mark.parametrize("k,pad", [(1, 0), (2, 0), (3, 0), (4, 0), (3, 1), (4, 1), (5, 0)])
def test_same_bits_as_the_permuted_product(handles, k, pad):
    h, r, c = handles
    g = torch.Generator(device="cuda")
    g.manual_seed(k)
    X = torch.rand(N, k, generator=g, device="cuda") - 0.5
    Y = torch.full((N, k + pad), 7.0, device="cuda")
    if k == 1:
        y = maxe.maxe_spmv(h, X[:, 0].contiguous())
        yp = maxe.maxe_spmv(h, X[:, 0][c.long()].contiguous(), permuted=True)
        assert torch.equal(y[r.long()], yp)
        return
    for _ in range(2):
        maxe.maxe_spmm(h, X, Y[:, :k])
    # the permuted product on 16-byte rows, as the x' and y' scratch have them
    kp = (k + 3) // 4 * 4
    Xp = torch.zeros(N, kp, device="cuda")[:, :k]
    Xp.copy_(X[c.long()])
    Yp = torch.zeros(N, kp, device="cuda")[:, :k]
    maxe.maxe_spmm(h, Xp, Yp, permuted=True)
    assert float((Y[r.long()][:, :k] - Yp).abs().max()) <= 2e-5
    assert bool((Y[:, k:] == 7.0).all())


def test_replayed_from_a_graph():
    A = W.poisson_uniform(4, N, 3.0, "f32", "cuda")
    r, c = maxe.maxe_build_permutation(2, N, 0), maxe.maxe_build_permutation(2, N, 1)
    h = maxe.from_csr(A, r, c, autotune=True)
    X = torch.rand(N, 4, device="cuda") - 0.5
    Y = torch.zeros(N, 4, device="cuda")
    Z = torch.zeros(N, 4, device="cuda")
    hs = torch.cuda.Stream()
    plain = maxe.from_csr(A, r, c)  # scatters in its epilogue
    maxe.maxe_spmm(plain, X, Z)
    maxe.maxe_spmm(h, X, Y)  # makes the scratch
    first = Y.clone()
    Y.zero_()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=hs):
        maxe.maxe_spmm(h, X, Y)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(Y, first)
    assert float((Y - Z).abs().max()) <= 2e-5
    h.close()
    plain.close()
