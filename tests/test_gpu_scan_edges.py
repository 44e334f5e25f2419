"""Scans on both sides of the sizes where their launches change: 8192 elements (one
CTA, or two launches) and 4096 tiles of 2048 (two launches, or three), the latter
through the P * ceil(k / 32) words of the column blocks' bitmaps."""
import numpy as np
import pytest

import oracle
from parity import assert_full_parity, run_gpu
from test_gpu_plan_sizes import banded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8191, 8192, 8193, 16384, 16385])
def test_one_cta_or_two_launches(n):
    rng = np.random.default_rng(n)
    A, B = banded(n, n, 3, rng, "i64"), banded(n, n, 2, rng, "i64")
    for P in (1, 32):                 # n column counts; 32 * ceil(n / 32) bitmap words
        assert_full_parity(run_gpu(A, B, P, 64), oracle.spgemm(A, B), f"n={n} P={P}")


@pytest.mark.parametrize("k", [(1 << 20) - 32, 1 << 20, (1 << 20) + 1])
def test_two_launches_or_three(k):
    """256 blocks: 4096 tiles of bitmap words less 256 words, exactly, and more."""
    rng = np.random.default_rng(7)
    A, B = banded(5000, k, 1, rng, "i64"), banded(k, 3000, 40, rng, "i64")
    assert_full_parity(run_gpu(A, B, 256, 4096), oracle.spgemm(A, B), f"k={k}")
