"""Edge probabilities are the float64 quotients rounded once to float32, also where a product kept to
48 bits would round the other way."""
import numpy as np
import pytest

from oracle import erc_oracle as O
from paper_2609_27209_gb300 import erc, synth

from ._gpu import build_both, host, to_dev

pytestmark = pytest.mark.gpu


def _kappa_of(w):
    """Curvatures, the largest of them 0, whose Eq. 8 weights sqrt(-kappa) + 1 are exactly w."""
    k = -((w - np.float32(1)) * (w - np.float32(1)))
    assert np.array_equal(np.sqrt(-k) + np.float32(1), w) and k.max() == 0
    return k


def _ring(m):
    """A graph of m edges (a ring)."""
    return m, np.arange(m, dtype=np.int32), (np.arange(m, dtype=np.int32) + 1) % m


# edge counts, and two weights in (2, 4) with 22 fraction bits, for which the product of the second with
# 1 / (1 + 2 (m - 3) + both) lies within 2^-48 of the middle between two float32 numbers
@pytest.mark.parametrize("m,pair,first", [
    (709, "0x1.68193dp+2", "0x1.b900dap+1"), (1582, "0x1.6dbf6cp+2", "0x1.3089840p+1"),
    (2694, "0x1.4927e4p+2", "0x1.409db0p+1"), (3168, "0x1.7030a2p+2", "0x1.83c6f6p+1"),
    (2284, "0x1.33c85bp+2", "0x1.43f954p+1")])
def test_edge_probabilities_hold_float64(m, pair, first):
    pair, first = float.fromhex(pair), float.fromhex(first)
    w = np.full(m, 2, np.float32)
    w[0], w[1], w[m - 1] = 1, first, pair - first
    total = w.astype(np.float64).sum()
    assert total == 1 + 2 * (m - 3) + pair  # exact in any order
    g, _ = build_both(*_ring(m))
    _, prob = erc.erc_sampling_probs(g, to_dev(_kappa_of(w)))
    np.testing.assert_array_equal(host(prob), (w.astype(np.float64) * (1.0 / total)).astype(np.float32))


@pytest.mark.parametrize("scale", [1e-30, 1.0, 1e30])
def test_edge_probabilities_over_the_range_of_weights(scale):
    """Against float64, from curvatures that leave every weight at 1 to weights of 1e15."""
    n, src, dst, _ = synth.random_connected(3000, 20000, seed=4, weighted=False)
    g, ref = build_both(n, src, dst)
    kappa = (np.random.default_rng(5).standard_normal(g.m) * scale).astype(np.float32)
    _, prob = erc.erc_sampling_probs(g, to_dev(kappa))
    k32 = np.maximum(-kappa + np.float32(2) * kappa.max(), np.float32(0))
    w = (np.sqrt(k32) + np.float32(1)).astype(np.float64)
    # the float32 weights' roundings are the kernel's own; the total's float64 sum has 53 bits
    np.testing.assert_allclose(host(prob), w / w.sum(), rtol=2.0 ** -24 + 2.0 ** -38)
    assert abs(host(prob).astype(np.float64).sum() - 1) < 2.0 ** -20
