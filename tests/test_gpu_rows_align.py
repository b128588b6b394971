"""SpMM with one row per lane group on X and Y rows of every alignment: the same
bits as on 16-byte rows, and nothing written outside the k columns."""
import pytest
import torch

from paper_2308_00106_gb300 import maxe
from paper_2308_00106_gb300 import workloads as W
from tests.gpu_common import check_all_rows_spmm, edge_matrix

pytestmark = pytest.mark.gpu


def _strided(n, k, ld, off, dtype, fill):
    return torch.full((n * ld + off,), fill, dtype=dtype, device="cuda")[off:].view(n, ld)[:, :k]


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("kind", ["ragged", "long_rows", "empty_runs"])
@pytest.mark.parametrize("k", [2, 3, 7, 8, 31, 33, 64])
def test_rows_any_alignment(kind, dtype, k):
    A = edge_matrix(kind, dtype, seed=8)
    h = maxe.from_csr(A.to("cuda"), spmm_rows=True)
    vt = torch.float64 if dtype == "f64" else torch.float32
    X0 = W.matrix_rhs(6, A.cols, k, "f64" if dtype == "f64" else "f32", "cuda")
    kp = (k + 3) // 4 * 4

    def product(xl, xo, yl, yo):
        X = _strided(A.cols, k, xl, xo, vt, float("nan"))
        X.copy_(X0)
        Y = _strided(A.rows, k, yl, yo, vt, 5.0)
        maxe.maxe_spmm(h, X, Y, permuted=True)
        whole = Y.as_strided((A.rows * yl,), (1,), yo)
        assert torch.all(whole.view(A.rows, yl)[:, k:] == 5.0)
        return Y

    Y = product(kp, 0, kp, 0)  # 16-byte rows on both sides
    rp, co, va = A.numpy()
    check_all_rows_spmm(Y.cpu().numpy(), rp, co, va, dtype, X0.cpu().numpy(), kind)
    for xl, xo, yl, yo in [(k, 0, k, 0), (kp, 0, kp + 1, 0), (kp + 2, 2, kp, 0), (kp + 1, 1, k + 1, 1), (kp, 4, k, 3)]:
        assert torch.equal(product(xl, xo, yl, yo), Y), (xl, xo, yl, yo)
    h.close()
