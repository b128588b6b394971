"""permute_csr's row ordering where bins are uneven or rows sit at the limits of a bucket: bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2308_00106_gb300 import maxe
from paper_2308_00106_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _matrix(kind, dtype):
    g = np.random.default_rng(11)
    cols = 200_000
    if kind == "lengths":  # empty, one, around the bins, the longest row of a bucket and the shortest long one
        lengths = np.concatenate([[0, 1, 2, 31, 32, 33, 0, 0, 2047, 2048, 1, 2049, 2048, 2048, 0], g.integers(0, 9, 3000)])
        parts = [g.choice(cols, n, replace=False) for n in lengths]
    elif kind == "clustered":  # half of a row's columns next to one another, the rest spread
        lengths = np.full(40, 1500)
        parts = [np.concatenate([1000 * i + np.arange(n // 2), g.choice(cols, n - n // 2)]) for i, n in enumerate(lengths)]
    elif kind == "repeated":  # one column many times: the old order has to stay
        lengths = g.integers(1, 700, 200)
        parts = [g.integers(0, 3, n) + 77 * i for i, n in enumerate(lengths)]
    else:  # "wide": more columns than a float counts exactly
        cols = 2**28 + 1
        lengths = g.integers(0, 300, 500)
        parts = [np.unique(np.concatenate([g.integers(0, cols, n), [cols - 1] * int(n > 0)]))[-n:] if n else [] for n in lengths]
        lengths = np.array([len(p) for p in parts])
    col = np.concatenate([np.asarray(p, dtype=np.int64) for p in parts])
    if kind != "repeated":  # unordered rows
        col = np.concatenate([g.permutation(np.asarray(p, dtype=np.int64)) for p in parts])
    rowptr = np.zeros(len(lengths) + 1, dtype=np.int64)
    rowptr[1:] = np.cumsum(lengths)
    val = torch.from_numpy(g.uniform(-1, 1, col.size)).to(W.DTYPES[dtype])
    return W.CSR(len(lengths), cols, torch.from_numpy(rowptr.astype(np.int32)), torch.from_numpy(col.astype(np.int32)),
                 val, dtype)


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("mode", ["none", "rows", "both"])
@pytest.mark.parametrize("kind", ["lengths", "clustered", "repeated", "wide"])
def test_rows_in_column_order(kind, mode, dtype):
    A = _matrix(kind, dtype)
    if kind == "wide" and mode == "both":
        pytest.skip("a column permutation of 2^28 columns takes the oracle minutes")
    r = maxe.maxe_build_permutation(3, A.rows, 0) if mode != "none" else None
    c = maxe.maxe_build_permutation(3, A.cols, 1) if mode == "both" else None
    h = maxe.from_csr(A.to("cuda"), r, c)
    rp, co, va = h.csr()[:3]
    host = lambda t: None if t is None else t.cpu().numpy()  # noqa: E731
    want = oracle.permute_csr(A.rows, A.cols, *A.numpy(), W.DTYPE_CODE[dtype], host(r), host(c))
    got = W.CSR(A.rows, A.cols, rp, co, va, dtype).numpy()
    for g, w in zip(got, want):
        np.testing.assert_array_equal(g, w)
    h.close()
