"""The Laplacian build at the edges of its sort and merge tiles and of its key digits: bit-exact
against the oracle, with self-loops, repeated pairs in both orientations and both policies."""
import numpy as np
import pytest

from paper_2609_27209_gb300 import erc, synth

from ._gpu import assert_graph_equal, build_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 2, 31, 2047, 2048, 2049, 4095, 4096, 4097, 8193, 20481])
@pytest.mark.parametrize("n", [1, 2, 15, 255, 256, 257, 5000, 70000])
def test_build_tile_edges(n, m):
    weighted = (m + n) % 2 == 0
    _, src, dst, w = synth.random_multigraph(n, m, seed=m + n, weighted=weighted)
    for policy in (erc.ERC_DUP_SUM, erc.ERC_DUP_FIRST):
        g, ref = build_both(n, src, dst, w, policy)
        assert_graph_equal(g, ref)


def test_build_long_runs_and_hubs():
    """One pair repeated 9,000 times (a run over several tiles), a hub of 3,000 neighbours (a row the
    degree sum gives to a whole warp), ids at the top of the range, most rows empty."""
    n = 100000
    hub = np.arange(n - 3001, n - 1, dtype=np.int32)
    src = np.concatenate([np.full(9000, 7, np.int32), np.full(3000, n - 1, np.int32)])
    dst = np.concatenate([np.full(9000, 3, np.int32), hub])
    w = synth.random_positive(src.size, 4, 0.5, 2.0)
    for weights in (None, w):
        for policy in (erc.ERC_DUP_SUM, erc.ERC_DUP_FIRST):
            g, ref = build_both(n, src, dst, weights, policy)
            assert_graph_equal(g, ref)


@pytest.mark.parametrize("m", [(2 << 20) - 1, 2 << 20, 342 * 6144 + 1])
def test_build_large_sort_tiles(m):
    """Around the input size from which the sort takes its large tiles."""
    _, src, dst, w = synth.random_multigraph(300000, m, seed=m, weighted=m % 2 == 0)
    g, ref = build_both(300000, src, dst, w)
    assert_graph_equal(g, ref)
