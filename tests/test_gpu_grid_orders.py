"""Orders that outrun the first graph of a run over the whole grid (L > 160):
slices narrowed, refills repeated, rounds added in chunks, the search in a
graph of its own, and the first graph captured anew with more rounds.  Caller
priorities against the CPU oracle, several runs on one handle."""
import numpy as np
import pytest

import oracle
from paper_1810_06800_gb300 import rsa, workloads

pytestmark = pytest.mark.gpu


def _keys(L, kind):
    if kind == "random":
        return workloads.permutation_keys(L, 7)
    return workloads.monotone_keys(L, descending=(kind == "descending"))


def _refills(lat):
    """Launches of the refill pass since the last call: one in the first graph
    of a run, one in each later chunk of rounds."""
    return rsa.rsa_kernel_stats(lat.h)["k_refill"][1]


def _run_is_exact(lat, L, k, keys):
    nj, nc = lat.run_keys(keys)
    wj, wc, _, acc = oracle.sample_keys(L, k, keys)
    assert (int(nj[0]), int(nc[0])) == (wj, wc)
    assert np.array_equal(lat.accepted(0), np.sort(acc))
    acc, _ = oracle.scan(L, k, keys)
    assert tuple(int(v[0]) for v in lat.contacts(1)) == oracle.contacts(L, k, acc)


@pytest.mark.parametrize("L,k", [(170, 2), (200, 8), (200, 40), (260, 129)])
def test_orders_on_the_grid(L, k):
    lat = rsa.Lattice(L, k)
    for kind in ("random", "monotone", "descending", "monotone"):
        _refills(lat)
        _run_is_exact(lat, L, k, _keys(L, kind))
        if kind == "monotone":
            assert _refills(lat) > 1  # more than the first graph ran
    # the same handle on seeds, with the longer first graph
    nj, nc = lat.run([5, 6])
    wj, wc = oracle.samples(L, k, [5, 6])
    assert np.array_equal(nj, wj.astype(np.uint32)) and np.array_equal(nc, wc.astype(np.uint32))
    lat.close()


@pytest.mark.parametrize("rounds", [1, 3, 64])
def test_rounds_per_check_past_the_first_graph(rounds):
    L, k = 200, 8
    lat = rsa.Lattice(L, k)
    rsa.rsa_set_rounds_per_check(lat.h, rounds)
    _refills(lat)
    _run_is_exact(lat, L, k, _keys(L, "monotone"))
    assert _refills(lat) > (2 if rounds < 64 else 1)
    lat.close()
