"""Deposition by priority slices against the CPU oracle where it can go wrong:
sides one off a bit word, k at the borders of its variants (block lines from
16 on, whole-warp window tests from 769, lanes per candidate at 129), lattices
barely longer than k, where windows and bins meet themselves round the torus,
and priority orders that fill the active set and the refilled list past their
capacities, so that slices are narrowed and refills repeated."""
import numpy as np
import pytest

import oracle
from paper_1810_06800_gb300 import rsa, workloads

pytestmark = pytest.mark.gpu


def _same(lat, sample, nj, nc, L, k, keys):
    wj, wc, _, acc = oracle.sample_keys(L, k, keys)
    assert (int(nj), int(nc)) == (wj, wc)
    assert np.array_equal(lat.accepted(sample), np.sort(acc))


@pytest.mark.parametrize("L,k", [(96, 15), (97, 16), (127, 17), (31, 16), (65, 33), (200, 96),
                                 (200, 97), (193, 128), (260, 129), (95, 95), (130, 127),
                                 (3, 2), (6, 5), (18, 17)])
def test_slice_shapes(L, k):
    seeds = [21, 22, 23]
    lat = rsa.Lattice(L, k)
    nj, nc = lat.run(seeds)
    nx, ny, nxy = lat.contacts(len(seeds))
    for i, s in enumerate(seeds):
        keys = oracle.keys(L, s)
        _same(lat, i, nj[i], nc[i], L, k, keys)
        acc, _ = oracle.scan(L, k, keys)
        assert (int(nx[i]), int(ny[i]), int(nxy[i])) == oracle.contacts(L, k, acc)
    lat.close()


@pytest.mark.parametrize("L,k", [(800, 768), (801, 769), (769, 769), (1100, 1055)])
def test_long_windows(L, k):
    seeds = [31, 32]
    lat = rsa.Lattice(L, k)
    nj, nc = lat.run(seeds)
    for i, s in enumerate(seeds):
        _same(lat, i, nj[i], nc[i], L, k, oracle.keys(L, s))
    lat.close()


@pytest.mark.parametrize("L,k", [(64, 8), (64, 2), (80, 33)])
@pytest.mark.parametrize("descending", [False, True])
def test_orders_that_overfill_a_slice(L, k, descending):
    keys = workloads.monotone_keys(L, descending=descending)
    lat = rsa.Lattice(L, k)
    nj, nc = lat.run_keys(keys)
    _same(lat, 0, nj[0], nc[0], L, k, keys)
    lat.close()
