"""Gradient-based permutations around 2^23 elements, where the halves' orders take different buckets:
bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2308_00106_gb300 import maxe

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1 << 23, (1 << 23) + 1, (1 << 23) + 3])
def test_halves_around_the_larger_buckets(n):
    h = np.random.default_rng(n).integers(0, 50, n).astype(np.int32)
    perm, pivot = maxe.maxe_gradient_permutation(torch.from_numpy(h).cuda(), 2308, 1)
    po, pvo = oracle.gradient_permutation(h, 2308, 1)
    np.testing.assert_array_equal(perm.cpu().numpy(), po)
    assert int(pivot.item()) == pvo
