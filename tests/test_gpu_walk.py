"""The row walk of the operator and the resident solver's dealt rows, at the sizes where they turn:
rows around the 4-, 8- and 16-neighbour steps and the heavy-row threshold, widths around the lane
groups and the 128-column slices, and a graph whose ids follow the degree.
"""
import numpy as np
import pytest
import torch

from oracle import erc_oracle as O
from paper_2609_27209_gb300 import erc, synth

from ._gpu import build_both, dev, host, to_dev
from .test_gpu_ops import _matvec_bound
from .test_gpu_solve import _check_R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("kc", [1, 20, 36, 64, 132, 300])
def test_apply_rows_of_every_step_length(kc, weighted):
    """Hub h has h neighbours of its own, h = 0..70 (0: an isolated node); the leaves have one."""
    lens = np.arange(71)
    src = np.repeat(lens, lens).astype(np.int32)
    dst = (71 + np.arange(src.size)).astype(np.int32)
    n = 71 + src.size
    w = synth.random_positive(src.size, 5) if weighted else None
    g, ref = build_both(n, src, dst, w)
    P = synth.random_block(n, kc, erc.padded_ld(kc), seed=kc)
    AP, pap = erc.erc_laplacian_apply(g, 1e-3, to_dev(P), kc, want_pap=True)
    Pk = P[:, :kc]
    APr = O.laplacian_matvec(ref, 1e-3, Pk.astype(np.float64))
    assert np.all(np.abs(host(AP)[:, :kc] - APr) <= _matvec_bound(ref, 1e-3, Pk))
    np.testing.assert_allclose(host(pap), np.einsum("ij,ij->j", Pk.astype(np.float64), APr),
                               rtol=2e-6)


@pytest.mark.parametrize("precond", [False, True])
@pytest.mark.parametrize("kc", [8, 36, 100])
def test_resident_solver_deals_rows_of_a_degree_ordered_graph(monkeypatch, kc, precond):
    """Ids by descending degree: the first of 152 contiguous ranges would hold a fifth of all
    neighbours, so the operator's rows are dealt out; the bars are those of the hub graphs."""
    monkeypatch.setenv("ERC_CG_MODE", "resident")
    n, src, dst, w = synth.chung_lu(8000, 2.2, 60000, "uniform_0.5_2", 3)
    g, ref = build_both(n, src, dst, w)
    Y = erc.erc_jl_rhs(g, 9, 256, 0, kc)
    fn = erc.erc_batched_pcg_timed if precond else erc.erc_batched_cg_timed
    X, iters, relres, st, _, path = fn(g, 1e-3, Y, kc, 1e-6)
    assert st == erc.ERC_OK and path == 1
    solve = O.batched_pcg if precond else O.batched_cg
    Xr, itr, _, _ = solve(ref, 1e-3, O.jl_rhs(ref, 9, 256, 0, kc), 1e-6)
    Rg = torch.zeros(g.m, device=dev())
    erc.erc_edge_resistance(g, X, kc, Rg)
    _check_R(host(Rg), O.edge_resistance(ref, Xr))
    assert np.all(np.abs(host(iters) - itr) <= 0.25 * itr + 3)
    assert np.all(host(relres) <= 4e-6)
