"""The samplers where node and edge count lie on either side of the count at which the scan tiles
grow from 2,048 to 8,192 entries (2^20), in a workspace of exactly the reported size: bytes after it
stay as they are, and the draws equal the oracle's."""
import numpy as np
import pytest
import torch

from oracle import sampler_oracle as S
from paper_2609_27209_gb300 import erc, synth

from ._gpu import build_both, dev, host, to_dev

pytestmark = pytest.mark.gpu

LARGE = 1 << 20


@pytest.mark.parametrize("n,m_in", [(900000, 2700000), (1200000, 1340000), (LARGE - 1, 1410000),
                                    (LARGE, 1390000), (LARGE + 1, 1300000)])
def test_sampler_stays_in_its_workspace(n, m_in):
    _, src, dst, _ = synth.random_multigraph(n, m_in, seed=n, weighted=False)
    g, ref = build_both(n, src, dst)
    assert (n < LARGE) != (g.m < LARGE)
    size = erc.lib().erc_sample_workspace_size(n, g.m, 5000)
    buf = torch.full((size + (1 << 20) + 1,), 0xA5, dtype=torch.uint8, device=dev())
    ws = buf[1:1 + size]  # the base as far from alignment as it can be
    rng = np.random.default_rng(n)
    for kind, count in ((erc.ERC_SAMPLE_NODES, n), (erc.ERC_SAMPLE_EDGES, g.m)):
        q = rng.random(count) ** 4
        q[count // 3: count // 3 + 20000] = 0.0  # runs of zero over whole tiles
        p = (q / q.sum()).astype(np.float32)
        for induced in (True, False):
            nodes, edges = erc.erc_sample_subgraph(g, kind, to_dev(p), 5000, 5, 3, induced=induced,
                                                   ws=ws)
            if kind == erc.ERC_SAMPLE_NODES:
                rn, re_ = S.sample_nodes(ref, p, 5000, 5, 3)
            else:
                rn, re_ = S.sample_edges(ref, p, 5000, 5, 3, induced=induced)
            np.testing.assert_array_equal(host(nodes), rn)
            np.testing.assert_array_equal(host(edges), re_)
            assert bool((buf[1 + size:] == 0xA5).all()) and int(buf[0]) == 0xA5
