"""Vector steps of the power iteration (maxe_vec_norm_gather, maxe_vec_dot_gather) against numpy in FP64."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# around one element, a block's round of loads (1024), two partials per thread (256 and 512 blocks), the largest split
SIZES = [1, 31, 1023, 1024, 1025, 256 * 1024, 256 * 1024 + 1, 512 * 1024 - 1, 512 * 1024 + 4097]


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("permuted", [False, True])
@pytest.mark.parametrize("n", SIZES)
def test_norm_and_dot_gather(n, permuted, dtype):
    from paper_2308_00106_gb300 import maxe

    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    w = torch.rand(n, generator=g, device="cuda", dtype=dtype) * 2 - 1
    u0 = torch.rand(n, generator=g, device="cuda", dtype=dtype) * 2 - 1
    Q = torch.randperm(n, generator=g, device="cuda").to(torch.int32) if permuted else None
    q = Q.cpu().numpy() if permuted else np.arange(n)
    wn, un = w.cpu().numpy().astype(np.float64), u0.cpu().numpy().astype(np.float64)
    scratch = torch.empty(514, dtype=torch.float64, device="cuda")
    out = torch.empty(1, dtype=torch.float64, device="cuda")
    maxe.maxe_vec_dot_gather(Q, u0, w, scratch, out)
    # an FP64 sum of n products, any order: error at most n u sum |terms|
    assert abs(out.item() - np.dot(un, wn[q])) <= n * 2.0 ** -52 * np.dot(np.abs(un), np.abs(wn[q]))
    u = torch.empty_like(w)
    maxe.maxe_vec_norm_gather(Q, w, u, scratch)
    want = wn[q] / np.sqrt(np.dot(wn, wn))
    # one rounding to the type, on top of a norm good to n u and three FP64 roundings
    eps = 2.0 ** -24 if dtype == torch.float32 else 0.0
    np.testing.assert_array_less(np.abs(u.cpu().numpy() - want), (eps + (n + 4) * 2.0 ** -52) * np.abs(want) + 1e-300)
