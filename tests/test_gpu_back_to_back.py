"""Products launched one behind the other without a gap, each reading what the one
before wrote and overwriting what it read: the same bits as with a
synchronisation after every launch."""
import pytest
import torch

from paper_2308_00106_gb300 import maxe
from paper_2308_00106_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STEPS = 40


def _run(h, V, permuted, wait):
    """STEPS products through two buffers, scaled into range by the matrix's values."""
    a, b = V.clone(), torch.empty_like(V)
    product = maxe.maxe_spmv if V.dim() == 1 else maxe.maxe_spmm
    for _ in range(STEPS):
        product(h, a, b, permuted=permuted)
        if wait:
            torch.cuda.synchronize()
        a, b = b, a
    return a


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("kernel", ["warp", "tuned", "xslice", "rows", "rows_odd"])
@pytest.mark.parametrize("permuted", [True, False])
@pytest.mark.parametrize("n", [300, 90_000])
def test_same_bits_with_and_without_waits(dtype, kernel, permuted, n):
    A = W.poisson_uniform(2, n, 6.0, dtype, "cuda")
    A.val = (A.val.float() * 0.2).to(A.val.dtype)
    flags = {"warp": {}, "tuned": {"autotune": True}, "xslice": {"xslice": True}, "rows": {"spmm_rows": True},
             "rows_odd": {"spmm_rows": True}}[kernel]
    h = maxe.from_csr(A, maxe.maxe_build_permutation(1, n, 0), maxe.maxe_build_permutation(1, n, 1), **flags)
    vt = torch.float64 if dtype == "f64" else torch.float32
    k = {"rows": 8, "rows_odd": 3}.get(kernel)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    V = torch.rand((n,) if k is None else (n, k), generator=g, device="cuda", dtype=vt) - 0.5
    ref = _run(h, V, permuted, True)
    assert bool(torch.isfinite(ref).all()) and bool((ref != 0).any())
    for _ in range(3):
        assert torch.equal(_run(h, V, permuted, False), ref)
    h.close()
