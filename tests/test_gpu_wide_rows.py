"""The operator on rows of 385 to 512 columns: the kernel for small blocks and the slices for large
ones, at the widths and node counts where one takes over from the other."""
import numpy as np
import pytest

from oracle import erc_oracle as O
from paper_2609_27209_gb300 import erc, synth

from ._gpu import build_both, host, to_dev
from .test_gpu_ops import _matvec_bound
from .test_gpu_resident_rows import _hubs, _two_steps

pytestmark = pytest.mark.gpu

EPS = 1e-3


def _check_apply(g, ref, kc, seed):
    P = synth.random_block(g.n, kc, erc.padded_ld(kc), seed=seed)
    AP, pap = erc.erc_laplacian_apply(g, EPS, to_dev(P), kc, want_pap=True)
    Pk = P[:, :kc]
    APr = O.laplacian_matvec(ref, EPS, Pk.astype(np.float64))
    assert np.all(np.abs(host(AP)[:, :kc] - APr) <= _matvec_bound(ref, EPS, Pk))
    np.testing.assert_allclose(host(pap), np.einsum("ij,ij->j", Pk.astype(np.float64), APr),
                               rtol=2e-6)


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("kc", [381, 384, 385, 449, 510, 512, 513])
def test_apply_rows_of_every_length(kc, weighted):
    n, src, dst = _hubs(4)
    w = synth.random_positive(src.size, 6, 0.5, 2.0) if weighted else None
    g, ref = build_both(n, src, dst, w)
    _check_apply(g, ref, kc, kc)


@pytest.mark.parametrize("n", [32767, 32768, 32769])
def test_apply_around_the_largest_small_block(n):
    """32,768 rows of 512 columns are 64 MB; one hub of 3,000 neighbours goes to a whole block."""
    _, src, dst, _ = synth.random_connected(n, 3 * n, seed=5, weighted=False)
    hub = np.arange(1, 3001, dtype=np.int32)
    g, ref = build_both(n, np.concatenate([src, np.zeros(3000, np.int32)]),
                        np.concatenate([dst, hub]))
    _check_apply(g, ref, 512, 1)


@pytest.mark.parametrize("precond", [False, True])
def test_two_steps_and_residual(monkeypatch, precond):
    """Bounds as in the resident solver's test of the same two steps."""
    monkeypatch.setenv("ERC_CG_MODE", "graph")
    n, src, dst = _hubs(4)
    g, ref = build_both(n, src, dst, synth.random_positive(src.size, 6, 0.5, 2.0))
    kc = 500
    Y = erc.erc_jl_rhs(g, 5, 512, 0, kc)
    fn = erc.erc_batched_pcg_timed if precond else erc.erc_batched_cg_timed
    X, iters, relres, st, _, path = fn(g, EPS, Y, kc, 1e-6, max_iter=2)
    assert path == 0 and st == erc.ERC_ERR_NOT_CONVERGED and np.all(host(iters) == 2)
    X64 = host(X).astype(np.float64)[:, :kc]
    Y64 = host(Y).astype(np.float64)[:, :kc]
    Xr = _two_steps(ref, Y64, precond)
    assert np.all(np.linalg.norm(X64 - Xr, axis=0) <= 1e-4 * np.linalg.norm(Xr, axis=0))
    rest = Y64 - O.laplacian_matvec(ref, EPS, X64)
    true = np.linalg.norm(rest, axis=0) / np.linalg.norm(Y64, axis=0)
    np.testing.assert_allclose(host(relres), true, rtol=1e-4)
