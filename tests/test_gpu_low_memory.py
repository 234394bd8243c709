"""A batch of small lattices on a GPU whose memory another allocator holds: the
workspaces of all blocks do not fit, those of some do."""
import numpy as np
import pytest

import oracle
from paper_1810_06800_gb300 import rsa

pytestmark = pytest.mark.gpu


def test_small_batch_in_little_free_memory():
    import torch
    L, k, seeds = 128, 4, list(range(1, 201))   # 1 MB a block, 152 blocks
    rsa.rsa_run_small(L, k, seeds[:1])          # kernels loaded
    rsa.rsa_mix_release()
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    free, _ = torch.cuda.mem_get_info()
    held = torch.empty(free - (100 << 20), dtype=torch.uint8, device="cuda")
    try:
        nj, nc = rsa.rsa_run_small(L, k, seeds)
    finally:
        del held
        torch.cuda.empty_cache()
        rsa.rsa_mix_release()
    wj, wc = oracle.samples(L, k, seeds)
    assert np.array_equal(nj, wj.astype(np.uint32)) and np.array_equal(nc, wc.astype(np.uint32))
