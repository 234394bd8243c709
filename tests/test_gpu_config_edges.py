"""Cluster sizes and winding directions on both sides of the line between one
block and several launches (8192 edges; k = 1 has 2 L^2), after runs of a
sample in one block and over the grid."""
import numpy as np
import pytest

import oracle
from paper_1810_06800_gb300 import rsa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,k", [(64, 1), (65, 1), (110, 2), (256, 12), (300, 16)])
def test_configuration_near_the_line(L, k):
    seeds = [4, 5]
    lat = rsa.Lattice(L, k)
    nj, nc = lat.run(seeds)
    for i in (1, 0, 1):
        acc, _ = oracle.scan(L, k, oracle.keys(L, seeds[i]))
        for m in (1, int(nc[i]) - 1, int(nc[i]), int(nj[i]) * 9 // 10, int(nj[i])):
            want, wx, wy = oracle.configuration(L, k, acc, m)
            assert np.array_equal(lat.cluster_sizes(i, m).astype(np.int64), want), (i, m)
            assert lat.wrap_dirs(i, m) == (wx, wy), (i, m)
    lat.close()
