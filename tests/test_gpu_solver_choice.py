"""The single-launch solver chosen where both fit: graphs on which the other one takes 15% to 90%
longer."""
import numpy as np
import pytest

from paper_2609_27209_gb300 import erc

from ._gpu import to_dev

pytestmark = pytest.mark.gpu

CLUSTER, RESIDENT = 2, 1


@pytest.mark.parametrize("n,per_node,kc,path", [
    (1000, 3, 16, CLUSTER), (3000, 12, 16, CLUSTER), (3000, 12, 128, CLUSTER),
    (3000, 3, 256, CLUSTER), (3000, 6, 256, CLUSTER), (10000, 3, 64, RESIDENT), (6000, 6, 128, RESIDENT),
    (10000, 12, 256, RESIDENT), (20000, 3, 16, RESIDENT)])
def test_solver_of_small_graphs(monkeypatch, n, per_node, kc, path):
    monkeypatch.delenv("ERC_CG_MODE", raising=False)
    rng = np.random.default_rng(n)
    ring = np.arange(n, dtype=np.int32)
    more = rng.integers(0, n, (2, (per_node - 1) * n)).astype(np.int32)
    src, dst = np.concatenate([ring, more[0]]), np.concatenate([(ring + 1) % n, more[1]])
    g = erc.erc_build_laplacian(n, to_dev(src), to_dev(dst.astype(np.int32)))
    Y = erc.erc_jl_rhs(g, 7, 256, 0, kc)
    assert erc.erc_batched_cg_timed(g, 1e-3, Y, kc, 1e-6)[5] == path
