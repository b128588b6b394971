"""Random permutations at the edges of the bucket split: one bucket, the shared-memory tile sizes, and
more buckets than are counted in shared memory."""
import numpy as np
import pytest

import oracle
from paper_2308_00106_gb300 import maxe

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2047, 2048, 2049, 8191, 8193, 1 << 22, (1 << 22) + 1, (1 << 24) + 1])
def test_build_permutation_bucket_edges(n):
    got = maxe.maxe_build_permutation(n ^ 0xABCDEF, n, n & 1).cpu().numpy()
    np.testing.assert_array_equal(got, oracle.build_permutation(n ^ 0xABCDEF, n, n & 1))
