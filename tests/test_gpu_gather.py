"""The row gather of X in original-space SpMM: on an identity matrix with permuted
rows and columns, Y = X to the bit for every row width, padding and alignment."""
import pytest
import torch

from paper_2308_00106_gb300 import maxe
from paper_2308_00106_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 33, 1025])
@pytest.mark.parametrize("k,ld,off", [(1, 1, 0), (2, 2, 0), (3, 4, 0), (4, 4, 0), (5, 8, 0), (7, 7, 0), (8, 9, 1),
                                      (4, 8, 2), (33, 36, 0), (64, 64, 0)])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_identity_returns_x(n, k, ld, off, dtype):
    vt = torch.float64 if dtype == "f64" else torch.float32
    idx = torch.arange(n + 1, dtype=torch.int32, device="cuda")
    A = W.CSR(n, n, idx, idx[:n].clone(), torch.ones(n, dtype=vt, device="cuda"), dtype)
    h = maxe.from_csr(A, maxe.maxe_build_permutation(3, n, 0), maxe.maxe_build_permutation(3, n, 1))
    g = torch.Generator(device="cuda")
    g.manual_seed(n + k)
    buf = torch.rand(n * ld + off, generator=g, dtype=vt, device="cuda")
    X = buf[off:].view(n, ld)[:, :k]
    assert torch.equal(maxe.maxe_spmm(h, X), X)
    h.close()
