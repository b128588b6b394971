"""The y' scratch of original-space products of large autotuned handles: made with the handle, never in a
call.  A product through it takes the kernel of the permuted product on rows of the same stride and copies
what that wrote, so the two agree bit for bit."""
import ctypes

import pytest
import torch

from paper_2308_00106_gb300 import maxe
from paper_2308_00106_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ORDER_BYTES = 30_000_000  # Y from which its rows are put in order later
VB = {"f64": 8, "f32": 4, "bf16": 4}


class CountingAllocator:
    """maxe_allocator over torch that records every call and refuses call number `refuse` (from 0)."""

    def __init__(self, refuse: int = -1):
        self.refuse, self.allocs, self.frees, self.live = refuse, [], [], {}
        A = maxe._Allocator
        self._fn = (A._fields_[0][1](self._alloc), A._fields_[1][1](self._free))
        self.struct = A(*self._fn, None)

    def _alloc(self, nbytes, ctx, stream):
        self.allocs.append(nbytes)
        if len(self.allocs) - 1 == self.refuse:
            return None
        t = torch.empty(max(int(nbytes), 1), dtype=torch.uint8, device="cuda")
        self.live[t.data_ptr()] = t
        return t.data_ptr()

    def _free(self, p, ctx, stream):
        self.frees.append(p)
        self.live.pop(p)


def _handle(n, dtype, al, seed=5):
    A = W.poisson_uniform(seed, n, 1.5, dtype, "cuda")
    r, c = maxe.maxe_build_permutation(seed, n, 0), maxe.maxe_build_permutation(seed, n, 1)
    csr = maxe._Csr(n, n, A.nnz, A.rowptr.data_ptr(), A.col.data_ptr(), A.val.data_ptr(), maxe.DTYPE_CODE[dtype])
    out = ctypes.c_void_p()
    maxe._check(maxe.load().maxe_permute_csr(ctypes.byref(csr), r.data_ptr(), c.data_ptr(), maxe.MAXE_AUTOTUNE,
                                             ctypes.byref(al.struct), maxe._stream(), ctypes.byref(out)), "permute")
    return maxe.Handle(out.value, n, n, A.nnz, maxe.DTYPE_CODE[dtype], keep=None), r.long(), c.long()


def _x(h, k, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.rand(h.cols, k, generator=g, device="cuda", dtype=h.vec_dtype) - 0.5


def _product(h, X):
    if X.shape[1] == 1:
        return maxe.maxe_spmv(h, X[:, 0].contiguous())[:, None]
    return maxe.maxe_spmm(h, X)


def _expected(h, r, c, X):
    """Y from the permuted product, its X and Y rows as the x' and y' scratch have them."""
    k = X.shape[1]
    y = torch.empty(h.rows, k, dtype=X.dtype, device="cuda")
    if k == 1:
        y[r, 0] = maxe.maxe_spmv(h, X[c, 0].contiguous(), permuted=True)
        return y
    Xp = torch.zeros(h.cols, (k + 3) // 4 * 4, dtype=X.dtype, device="cuda")[:, :k]
    Xp.copy_(X[c])
    Yp = torch.empty(h.rows, 16 // X.element_size(), dtype=X.dtype, device="cuda")[:, :k]
    y[r] = maxe.maxe_spmm(h, Xp, Yp, permuted=True)
    return y


@pytest.mark.parametrize("dtype,ks", [("f32", (1, 4, 1, 2, 3, 4)), ("bf16", (1, 4, 3)), ("f64", (1, 2, 1))])
def test_no_call_allocates_and_every_k_has_the_permuted_bits(dtype, ks):
    n = ORDER_BYTES // VB[dtype] + 1  # k = 1 just past the line, so all of them
    al = CountingAllocator()
    h, r, c = _handle(n, dtype, al)
    assert 16 * n in al.allocs
    made, freed = len(al.allocs), len(al.frees)
    for i, k in enumerate(ks):
        X = _x(h, k, i)
        assert torch.equal(_product(h, X), _expected(h, r, c, X)), k
    assert (len(al.allocs), len(al.frees)) == (made, freed)
    h.close()
    assert not al.live


@pytest.mark.parametrize("k", [2, 3])
@pytest.mark.parametrize("past", [0, 1])
def test_rows_around_the_line(k, past):
    n = ORDER_BYTES // (4 * k) + past
    h, r, c = _handle(n, "f32", CountingAllocator())
    X = _x(h, k, k)
    Y = _product(h, X)
    # the scattering kernel may sum in another order: rows hold at most 14 entries (Poisson, mean 1.5, 1e7
    # rows: P < 1e-3), |a| <= 1, |x| <= 1/2, so two orders differ by at most 2 * 15 * 2^-24 * 7 < 1.3e-5
    assert float((Y - _expected(h, r, c, X)).abs().max()) <= 1.3e-5
    h.close()


def test_a_graph_of_spmv_survives_wider_products():
    n = ORDER_BYTES // 4 + 1
    al = CountingAllocator()
    h, _, _ = _handle(n, "f32", al)
    X, X4 = _x(h, 1, 1), _x(h, 4, 2)
    x, y = X[:, 0].contiguous(), torch.zeros(n, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):  # no product before it
        maxe.maxe_spmv(h, x, y)
    graph.replay()
    first = y.clone()
    assert torch.equal(first, maxe.maxe_spmv(h, x))
    maxe.maxe_spmm(h, X4)
    others = [torch.full((n,), 3.0, device="cuda") for _ in range(8)]  # would take any freed block
    y.zero_()
    graph.replay()
    assert torch.equal(y, first)
    assert all(bool((t == 3.0).all()) for t in others)
    h.close()


@pytest.mark.parametrize("unit", [16, 4])
def test_without_the_memory_rows_are_scattered(unit):
    """Neither the scratch (16 bytes a row) nor the inverse permutation (4) is needed for the result."""
    n = ORDER_BYTES // 4 + 12_345
    al = CountingAllocator()
    _handle(n, "f32", al)[0].close()
    al = CountingAllocator(max(i for i, b in enumerate(al.allocs) if b == unit * n))  # the last of that size
    h, r, c = _handle(n, "f32", al)
    X = _x(h, 1, 3)
    assert torch.equal(_product(h, X), _expected(h, r, c, X))
    h.close()
    assert not al.live
