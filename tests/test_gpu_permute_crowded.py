"""permute_csr on rows whose columns crowd into few of their bins: bit-exact against the oracle on both sides
of the rule that sorts such a bucket instead, and no time that grows with the square of a row."""
import numpy as np
import pytest
import torch

import oracle
from paper_2308_00106_gb300 import maxe
from paper_2308_00106_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _crowded(lengths, crowd, cols, dtype, seed=17):
    """Unordered rows: `crowd` of a row's columns next to one another, the others spread over all."""
    g = np.random.default_rng(seed)
    parts = []
    for i, n in enumerate(lengths):
        near = 7 * i + np.arange(min(n, crowd))
        far = cols // 2 + g.choice(cols // 2, n - near.size, replace=False)
        parts.append(g.permutation(np.concatenate([near, far])))
    rowptr = np.concatenate([[0], np.cumsum(lengths)])
    col = np.concatenate(parts).astype(np.int32)
    val = torch.from_numpy(g.uniform(-1, 1, col.size)).to(W.DTYPES[dtype])
    return W.CSR(len(lengths), cols, torch.from_numpy(rowptr.astype(np.int32)), torch.from_numpy(col), val, dtype)


# the rule is at 250,000 comparisons: a bin of 500 entries; 12 rows of 145 in a bucket; and buckets of 4095 entries
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("identity", [False, True])
@pytest.mark.parametrize("lengths,crowd", [([2048] * 9, 490), ([2048] * 9, 505), ([2048] * 9, 2047),
                                           ([2047, 2048] * 5, 500), ([180] * 300, 144), ([1] * 2047 + [2048] * 3, 2048),
                                           ([3] * 700 + [1025] * 40 + [0] * 5, 1024)])
def test_crowded_rows(lengths, crowd, identity, dtype):
    A = _crowded(lengths, crowd, 4_000_000, dtype)
    c = torch.arange(A.cols, dtype=torch.int32, device="cuda") if identity else None
    r = maxe.maxe_build_permutation(3, A.rows, 0)
    h = maxe.from_csr(A.to("cuda"), r, c)
    want = oracle.permute_csr(A.rows, A.cols, *A.numpy(), W.DTYPE_CODE[dtype], r.cpu().numpy(),
                              None if c is None else c.cpu().numpy())
    for got, w in zip(W.CSR(A.rows, A.cols, *h.csr()[:3], dtype).numpy(), want):
        np.testing.assert_array_equal(got, w)
    h.close()


def test_one_column_repeated():
    """All entries of a bucket in one bin and one column: the old order stays."""
    n, rows = 2048, 6
    val = torch.rand(n * rows, device="cuda")
    A = W.CSR(rows, 10, torch.arange(rows + 1, dtype=torch.int32, device="cuda") * n,
              torch.full((n * rows,), 7, dtype=torch.int32, device="cuda"), val, "f32")
    h = maxe.from_csr(A)
    assert torch.equal(h.csr()[2], val)
    h.close()


def test_a_band_takes_no_quadratic_time():
    """Rows of 2000 neighbouring columns of 2^26: under the identity all of a row falls into one bin, under a
    random permutation hardly two entries do.  Ranked within that bin they took over twenty times as long."""
    rows, n, cols = 12_500, 2000, 1 << 26
    col = (torch.arange(rows, device="cuda").view(-1, 1) * 8 + torch.arange(n, device="cuda")).int().reshape(-1)
    A = W.CSR(rows, cols, torch.arange(rows + 1, dtype=torch.int32, device="cuda") * n, col.contiguous(),
              torch.ones(rows * n, device="cuda"), "f32")

    def ms(cperm):
        best = 1e9
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            h = maxe.from_csr(A, None, cperm)
            b.record()
            torch.cuda.synchronize()
            h.close()
            best = min(best, a.elapsed_time(b))
        return best

    random = ms(maxe.maxe_build_permutation(5, cols, 1))
    assert ms(torch.arange(cols, dtype=torch.int32, device="cuda")) <= 6 * random
