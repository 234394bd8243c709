"""First wrap at a k-mer with many earlier neighbours.  All its edges have its
priority for time, so the window of the search comes down to one time and still
holds more edges than its last stage takes one by one (32) or keeps in shared
memory (4096).  n_c does not depend on the number of edges (Sec. II.D)."""
import numpy as np
import pytest

import oracle
from paper_1810_06800_gb300 import rsa

pytestmark = pytest.mark.gpu


def _keys(L, first, rng_seed):
    """Priorities that try `first` in the given order, then the rest at random."""
    rng = np.random.default_rng(rng_seed)
    keys = np.empty(2 * L * L, dtype=np.uint64)
    rest = np.setdiff1d(np.arange(keys.size), first)
    keys[first] = np.arange(1, len(first) + 1)
    keys[rest] = rng.permutation(rest.size) + len(first) + 1
    return keys


def _comb(L):
    """k = L - 1: horizontal k-mers on k rows leave column 0 free, then a
    vertical one fills it and meets both ends of each, 2 k edges."""
    return [y * L + 1 for y in range(L - 1)] + [L * L]


# rows of k-mers up to column 63, one from column 65 on, and the vertical one
# between them: 41 edges, one of them closes the wrap
FORTY = [y * 129 for y in range(40)] + [65, 129 * 129 + 64]


@pytest.mark.parametrize("L,k,first", [
    pytest.param(41, 40, _comb(41), id="one block"),
    pytest.param(129, 64, FORTY, id="one block, 41 edges"),
    pytest.param(201, 200, _comb(201), id="grid"),
    pytest.param(2050, 2049, _comb(2050), id="grid, more edges than the last window holds"),
])
def test_wrap_at_a_kmer_of_many_edges(L, k, first):
    keys = _keys(L, first, 3)
    lat = rsa.Lattice(L, k)
    nj, nc = lat.run_keys(keys)
    wj, wc, _, acc = oracle.sample_keys(L, k, keys)
    assert wc == len(first)
    assert (int(nj[0]), int(nc[0])) == (wj, wc)
    assert np.array_equal(lat.accepted(0), np.sort(acc))
    lat.close()
