"""The largest graphs that the resident solver takes: what its rows need in shared memory leaves it the
sizes for which it is the fastest solver."""
import pytest

from paper_2609_27209_gb300 import erc, synth

from ._gpu import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,kc,weighted", [(245000, 16, True), (124800, 32, True),
                                           (124800, 32, False), (62700, 64, True),
                                           (31400, 128, True), (15000, 256, True)])
def test_resident_solver_takes_graphs_up_to(monkeypatch, n, kc, weighted):
    """r and Ap of n x kc float32 values fill the 227 KB of 152 SMs at n kc = 4.42 million; these sizes
    lie 9% to 13% below that."""
    monkeypatch.setenv("ERC_CG_MODE", "resident")
    src, dst = synth.random_multigraph(n, 2 * n, seed=n, weighted=False)[1:3]
    w = synth.random_positive(src.size, 3, 0.5, 2.0) if weighted else None
    g = erc.erc_build_laplacian(n, to_dev(src), to_dev(dst), to_dev(w))
    Y = erc.erc_jl_rhs(g, 5, 256, 0, kc)
    _, _, relres, st, _, path = erc.erc_batched_cg_timed(g, 1e-3, Y, kc, 1e-3)
    assert st == erc.ERC_OK and path == 1 and float(relres.max()) <= 2e-3
