"""Counts and entropy where the histogram takes more than the smallest run of entries per CTA."""
import numpy as np
import pytest
import torch

from paper_2308_00106_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ROWS, COLS = 200_003, 150_001  # 50 entries a row: 10 M entries, above one resident wave of the smallest runs


@pytest.fixture(scope="module")
def handle():
    from paper_2308_00106_gb300 import maxe

    A = W.poisson_uniform(7, ROWS, 50.0, "f32", "cuda", cols=COLS)
    h = maxe.from_csr(A)
    yield A, h
    h.close()


# one bin, the benches' grid, one row bin with as many column bins as fit a CTA and one more, many row bins, rows by columns
@pytest.mark.parametrize("grid", [(1, 1), (64, 64), (1, 8192), (1, 8193), (2, 4096), (600, 13), (ROWS, 1), (3, COLS)])
def test_counts_and_entropy(handle, grid):
    from paper_2308_00106_gb300 import maxe

    A, h = handle
    gr, gc = grid
    H, counts = maxe.maxe_nnz_entropy(h, gr, gc)
    rp = A.rowptr.long()
    rows = torch.repeat_interleave(torch.arange(ROWS, device="cuda"), rp[1:] - rp[:-1])
    want = torch.bincount((rows * gr // ROWS) * gc + A.col.long() * gc // COLS, minlength=gr * gc).cpu().numpy()
    np.testing.assert_array_equal(counts.cpu().numpy().reshape(-1), want)
    p = want[want > 0] / A.nnz
    ref = -(p * np.log2(p)).sum()
    # terms are good to a few ulp, the sum of n of them to n u of their sum (which is H)
    assert abs(H - ref) <= (p.size + 8) * 2.0 ** -52 * max(ref, 1.0)
