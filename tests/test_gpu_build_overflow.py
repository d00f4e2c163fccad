"""Degrees and merged weights past the largest float32 are infinite, as the rounded float64 sum is."""
import numpy as np
import pytest

from paper_2609_27209_gb300 import erc

from ._gpu import build_both, host

pytestmark = pytest.mark.gpu

MAX = np.finfo(np.float32).max


@pytest.mark.parametrize("neighbours", [2, 7, 8, 9, 40, 256, 257, 3000])
@pytest.mark.parametrize("big", [1, 2, 17])
def test_degree_past_the_largest_float(neighbours, big):
    """A star whose hub has `big` edges of the largest weight among small ones: its degree is the
    largest float with one of them, infinite from two on; no other degree is touched."""
    n = neighbours + 1
    src = np.zeros(neighbours, np.int32)
    dst = np.arange(1, n, dtype=np.int32)
    w = np.ones(neighbours, np.float32)
    w[np.linspace(0, neighbours - 1, min(big, neighbours)).astype(int)] = MAX
    with np.errstate(over="ignore"):
        g, ref = build_both(n, src, dst, w)
        expect = np.float32(w.astype(np.float64).sum())
    assert np.isinf(expect) == (min(big, neighbours) > 1)
    assert host(g.deg)[0] == expect
    np.testing.assert_array_equal(host(g.deg), ref["deg"])


@pytest.mark.parametrize("policy", [erc.ERC_DUP_SUM, erc.ERC_DUP_FIRST])
def test_merged_weight_past_the_largest_float(policy):
    """A pair given three times with the largest weight, in a row of 300 other neighbours."""
    n = 302
    src = np.concatenate([np.zeros(300, np.int32), np.full(3, 301, np.int32)])
    dst = np.concatenate([np.arange(1, 301, dtype=np.int32), np.zeros(3, np.int32)])
    w = np.concatenate([np.full(300, 0.5, np.float32), np.full(3, MAX, np.float32)])
    with np.errstate(over="ignore"):
        g, ref = build_both(n, src, dst, w, policy)
    merged = np.inf if policy == erc.ERC_DUP_SUM else MAX
    assert host(g.deg)[301] == merged
    np.testing.assert_array_equal(host(g.ew), ref["ew"])
    np.testing.assert_array_equal(host(g.deg), ref["deg"])
