"""Workspace of shapes with about 2^14 k-mers, past the last that a sample in one
block could hold: nothing is set aside there for a search in one block.  Host
arithmetic only."""
import pytest

from paper_1810_06800_gb300 import build, rsa


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("L,k", [(256, 4), (512, 16), (1024, 64), (400, 10)])
def test_longer_kmers_need_no_more(L, k):
    # fewer k-mers and edges, shorter lists
    assert rsa.rsa_workspace_bytes(L, k, 1) <= rsa.rsa_workspace_bytes(L, k - 1, 1)


def test_static_array_holds_twenty_samples():
    # 64 MiB of rsa_run_static at L = 256, k = 4: 3.4 MB a sample
    assert rsa.rsa_workspace_bytes(256, 4, 20) <= 64 << 20
