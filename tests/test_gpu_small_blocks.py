"""rsa_run_small with more samples than SMs: the library's choice of the block
size and of several blocks per SM (256, 512 and 1024 threads here)."""
import numpy as np
import pytest

import oracle
from paper_1810_06800_gb300 import rsa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,k", [(1, 1), (16, 2), (40, 4), (128, 128), (64, 4)])
def test_more_samples_than_sms(L, k):
    seeds = list(range(100, 800))
    nj, nc = rsa.rsa_run_small(L, k, seeds)
    wj, wc = oracle.samples(L, k, seeds)
    assert np.array_equal(nj, wj.astype(np.uint32)) and np.array_equal(nc, wc.astype(np.uint32))
