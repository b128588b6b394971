"""MAXE_SPMM_ROWS_PF acts at every k.  Results do not depend on it, its time does: on the permuted 4096 x 4096
Laplacian in FP64 each prefetched row of four columns costs a line that leaves L2 unused (1932 us without,
2750 us with it)."""
import pytest
import torch

from paper_2308_00106_gb300 import maxe
from paper_2308_00106_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_the_prefetch_flag_acts_below_sixteen_columns():
    A = W.laplacian5(4096, "f64", "cuda")
    r, c = maxe.maxe_build_permutation(1, A.rows, 0), maxe.maxe_build_permutation(1, A.cols, 1)
    X = torch.rand(A.cols, 4, dtype=torch.float64, device="cuda")
    times, results = [], []
    for pf in (False, True):
        h = maxe.from_csr(A, r, c, spmm_rows=True, spmm_rows_pf=pf)
        assert h.spmm_rows_prefetch() == pf
        Y = torch.empty(A.rows, 4, dtype=torch.float64, device="cuda")
        best = 1e9
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            maxe.maxe_spmm(h, X, Y, permuted=True)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        times.append(best)
        results.append(Y)
        h.close()
    assert torch.equal(*results)
    assert times[1] > 1.15 * times[0]
