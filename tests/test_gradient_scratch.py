"""The workspace that the gradient-based permutation asks for holds either half of the deck (CPU: the
allocator records each request and refuses it, so nothing is launched).  The workspace of an order is not
monotone in its length -- above 2^22 indices the buckets get larger and fewer -- so the longer half's need
not cover the shorter one's."""
import ctypes

import pytest

from paper_2308_00106_gb300 import build as B
from paper_2308_00106_gb300 import maxe

ALIGNED = 256  # a stand-in for a device address: no request succeeds, so it is never read


def _requests(call):
    """Bytes of every allocation that `call(allocator)` asks for; all are refused."""
    asked = []
    A = maxe._Allocator
    alloc = A._fields_[0][1](lambda nbytes, ctx, stream: asked.append(nbytes))
    free = A._fields_[1][1](lambda ptr, ctx, stream: None)
    assert call(ctypes.byref(A(alloc, free, None))) == maxe.MAXE_ERR_OOM
    return asked


@pytest.fixture(scope="module")
def lib():
    B.build()
    return maxe.load()


def _order_bytes(lib, n):
    return _requests(lambda al: lib.maxe_build_permutation(1, n, 0, ALIGNED, al, None))[0]


@pytest.mark.parametrize("n", [4096, 4097, 8191, 1 << 20, (1 << 23) - 1, 1 << 23, (1 << 23) + 1, (1 << 23) + 2,
                               (1 << 24) + 1, (1 << 26) + 1, (1 << 30) + 1])
def test_workspace_holds_both_halves(lib, n):
    order, workspace, _ = _requests(
        lambda al: lib.maxe_gradient_permutation(ALIGNED, n, 1, 0, ALIGNED, None, al, None))
    assert order == 4 * n
    half = (n + 1) // 2
    assert workspace >= max(_order_bytes(lib, half), _order_bytes(lib, n - half))
