"""Edges of the steps and tiles of the right-hand side, the edge distances and the samplers."""
import numpy as np
import pytest
import torch

from oracle import erc_oracle as O
from oracle import sampler_oracle as S
from paper_2609_27209_gb300 import erc, synth

from ._gpu import build_both, host, to_dev
from .test_gpu_ops import U32, _rhs_bound

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("K,c0,kc", [(16, 12, 1), (64, 28, 13), (200, 100, 100), (400, 124, 132),
                                     (700, 116, 520), (1100, 60, 1024)])
def test_jl_rhs_spans_sign_blocks(K, c0, kc, weighted):
    """Batches that start inside a 128-column sign block and span up to nine, rows longer and
    shorter than a lane group."""
    n, src, dst, w = synth.chung_lu(600, 2.2, 6000, "uniform_0.5_2" if weighted else "unit", 8)
    g, ref = build_both(n, src, dst, w)
    Y = host(erc.erc_jl_rhs(g, 99, K, c0, kc))
    Yr = O.jl_rhs(ref, 99, K, c0, kc)
    assert np.all(Y[:, kc:] == 0)
    assert np.all(np.abs(Y[:, :kc] - Yr) <= _rhs_bound(ref, K)[:, None] + 1e-30)


@pytest.mark.parametrize("m", [1, 3, 4, 5, 31, 33, 1022])
@pytest.mark.parametrize("kc", [3, 20, 50, 128, 200, 400, 1000])
def test_edge_resistance_step_edges(m, kc):
    """Edge counts around the steps of a segment, runs of equal first endpoints across steps (a star
    with a path through its leaves)."""
    n = m + 2
    hub = np.zeros((m + 1) // 2, np.int32)
    src = np.concatenate([hub, np.arange(1, 1 + m - hub.size, dtype=np.int32)])
    dst = np.concatenate([1 + np.arange(hub.size, dtype=np.int32),
                          2 + np.arange(m - hub.size, dtype=np.int32)])
    g, ref = build_both(n, src, dst)
    X = synth.random_block(n, kc, erc.padded_ld(kc), seed=kc)
    R0 = synth.random_positive(g.m, seed=3)
    R = to_dev(R0.copy())
    erc.erc_edge_resistance(g, to_dev(X), kc, R)
    Rr = R0.astype(np.float64) + O.edge_resistance(ref, X[:, :kc].astype(np.float64))
    np.testing.assert_allclose(host(R), Rr, rtol=(kc + 8) * U32)


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n", [2, 63, 64, 65, 8191, 8192, 8193, 20500])
def test_sampler_tile_edges(n, shift):
    """Node and edge draws over counts around the search steps and scan tiles, with runs of zero
    probability over whole steps and tiles; shift: probabilities off 16-byte alignment."""
    _, src, dst, _ = synth.random_connected(n, 3 * n, seed=n, weighted=False)
    g, ref = build_both(n, src, dst)
    rng = np.random.default_rng(n)
    for kind, count in ((erc.ERC_SAMPLE_NODES, n), (erc.ERC_SAMPLE_EDGES, g.m)):
        q = rng.random(count) ** 4
        q[count // 3: count // 3 + min(count // 2, 9000)] = 0.0
        p = (q / q.sum()).astype(np.float32)
        dev_p = torch.zeros(count + shift, device="cuda:0")[shift:]
        dev_p.copy_(to_dev(p))
        for budget, induced in ((1, True), (700, True), (700, False)):
            nodes, edges = erc.erc_sample_subgraph(g, kind, dev_p, budget, 5, 3, induced=induced)
            if kind == erc.ERC_SAMPLE_NODES:
                rn, re_ = S.sample_nodes(ref, p, budget, 5, 3)
            else:
                rn, re_ = S.sample_edges(ref, p, budget, 5, 3, induced=induced)
            np.testing.assert_array_equal(host(nodes), rn)
            np.testing.assert_array_equal(host(edges), re_)
