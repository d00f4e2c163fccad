"""The Laplacian build at the edges of the sort's large tiles (2,560 keys, from 2^21 keys on)."""
import pytest

from paper_2609_27209_gb300 import synth

from ._gpu import assert_graph_equal, build_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [820 * 2560 - 1, 820 * 2560, 820 * 2560 + 1])
def test_build_large_tile_edges(m):
    assert m >= 2 << 20
    _, src, dst, w = synth.random_multigraph(300000, m, seed=m, weighted=m % 2 == 0)
    g, ref = build_both(300000, src, dst, w)
    assert_graph_equal(g, ref)
