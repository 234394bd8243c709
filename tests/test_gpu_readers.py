"""Several threads that read one finished handle: each gets the whole result,
also when they are the first to read it (include/rsa.h, conventions)."""
import threading

import numpy as np
import pytest

from paper_1810_06800_gb300 import rsa

pytestmark = pytest.mark.gpu


def test_threads_read_one_handle():
    # 38 MB of sample states: freed ones are unmapped at once
    n = 300_000
    L, k = 8, 4
    lat = rsa.Lattice(L, k)
    for run in range(4):
        seeds = np.arange(run * n, (run + 1) * n, dtype=np.uint64)
        rsa.rsa_run_seeds(lat.h, seeds)
        gate = threading.Barrier(4)
        got = [None] * 4

        def read(i):
            gate.wait()
            nj, nc = rsa.rsa_results(lat.h, n)
            got[i] = [nj, nc, *lat.contacts(n), rsa.rsa_sample_stats(lat.h, n)["edges"]]

        threads = [threading.Thread(target=read, args=(i,)) for i in range(4)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        want = [*rsa.rsa_results(lat.h, n), *lat.contacts(n),
                rsa.rsa_sample_stats(lat.h, n)["edges"]]
        for values in got:
            assert values is not None
            for a, b in zip(values, want):
                assert np.array_equal(a, b)
    lat.close()
