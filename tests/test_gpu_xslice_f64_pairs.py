"""FP64 x-sliced SpMV on CTA pairs: taken where the library chooses (even column
halves, one wave of tiles), against the FP64 oracle on every row."""
import pytest
import torch

from paper_2308_00106_gb300 import maxe
from paper_2308_00106_gb300 import workloads as W
from tests.gpu_common import check_all_rows

pytestmark = pytest.mark.gpu


def _handle(A, seed):
    return maxe.from_csr(A, maxe.maxe_build_permutation(seed, A.rows, 0), maxe.maxe_build_permutation(seed, A.cols, 1),
                         xslice=True)


@pytest.mark.parametrize("n", [60_000, 199_999])
@pytest.mark.parametrize("kind", ["powerlaw", "poisson"])
def test_pairs_against_oracle(kind, n):
    if kind == "powerlaw":
        A = W.powerlaw(3, n=n, dtype="f64", device="cuda")
    else:
        A = W.poisson_uniform(3, n, 30.0, "f64", "cuda")
    h = _handle(A, 5)
    assert h.xslice() and h.xslice_pairs()
    x = W.vector(7, A.cols, "f64", "cuda")
    y = maxe.maxe_spmv(h, x)
    rp, co, va = A.to("cpu").numpy()
    check_all_rows(y.cpu().numpy(), rp, co, va, "f64", x.cpu().numpy(), kind)
    assert torch.equal(maxe.maxe_spmv(h, x), y)
    h.close()


@pytest.mark.parametrize("n,lam", [(1_400_000, 3.0), (4096, 20.0)])
def test_single_ctas_where_pairs_do_not_fit(n, lam):
    """More rows than one wave of pairs has accumulators for; a matrix of one column slice."""
    A = W.poisson_uniform(4, n, lam, "f64", "cuda")
    h = _handle(A, 6)
    assert h.xslice() and not h.xslice_pairs()
    x = W.vector(8, A.cols, "f64", "cuda")
    rp, co, va = A.to("cpu").numpy()
    check_all_rows(maxe.maxe_spmv(h, x).cpu().numpy(), rp, co, va, "f64", x.cpu().numpy())
    h.close()
