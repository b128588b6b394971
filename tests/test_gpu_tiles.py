"""The staged-tile SpMV against the FP64 oracle, every row within the rounding
bound of its terms: rows across tile ends, rows longer than a lane group's share
and than a tile, empty rows, one entry a row, in both spaces."""
import numpy as np
import pytest
import torch

from paper_2308_00106_gb300 import maxe
from paper_2308_00106_gb300 import workloads as W
from tests.gpu_common import check_all_rows, edge_matrix, oracle_permuted

pytestmark = pytest.mark.gpu


def _matrix(kind, dtype):
    if kind == "tile_ends":  # rows of 1984, 2041..2056 and 32 G + 1 entries among short ones
        lengths = np.random.default_rng(5).integers(0, 9, 4000)
        lengths[[7, 900, 901, 1800, 2500, 3999]] = [1984, 2041, 2048, 2049, 2056, 33]
        return W.from_lengths(5, lengths, 6000, dtype)
    if kind == "many_tiles":  # more entries than eight full tiles per SM
        return W.from_lengths(6, np.random.default_rng(6).integers(0, 12, 480_000), 70_001, dtype)
    return edge_matrix(kind, dtype, seed=4)


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("kind", ["one", "ragged", "empty_runs", "unit_rows", "long_rows", "rect_wide", "rect_tall",
                                  "tile_ends", "many_tiles"])
def test_tiles_against_oracle(kind, dtype):
    A = _matrix(kind, dtype)
    rperm = maxe.maxe_build_permutation(9, A.rows, 0)
    cperm = maxe.maxe_build_permutation(9, A.cols, 1)
    h = maxe.from_csr(A.to("cuda"), rperm, cperm, autotune=True)
    x = W.vector(4, A.cols, "f64" if dtype == "f64" else "f32", "cuda")
    rp, co, va = A.numpy()
    y = maxe.maxe_spmv_tiles(h, x)
    check_all_rows(y.cpu().numpy(), rp, co, va, dtype, x.cpu().numpy(), kind)
    assert torch.equal(maxe.maxe_spmv_tiles(h, x), y)
    xp = x[cperm.long()].contiguous()
    yp = maxe.maxe_spmv_tiles(h, xp, permuted=True)
    assert torch.equal(yp, y[rperm.long()])
    h.close()


def test_handles_without_tiles_refuse():
    for A, tune in [(edge_matrix("ragged"), False), (edge_matrix("empty_nnz"), True)]:
        h = maxe.from_csr(A.to("cuda"), autotune=tune)
        with pytest.raises(maxe.MaxeError):
            maxe.maxe_spmv_tiles(h, torch.zeros(A.cols, device="cuda"))
        h.close()
