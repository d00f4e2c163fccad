"""The resident solver's gathers at the lengths and widths where its steps turn: rows of 0 to 40
neighbours side by side in a warp (steps of 4, 8 and 16, and rows given to whole blocks), row groups
of 4 to 32 lanes with and without spare ones, rows of two quads a lane."""
import numpy as np
import pytest

from oracle import erc_oracle as O
from paper_2609_27209_gb300 import erc, synth

from ._gpu import build_both, host

pytestmark = pytest.mark.gpu

EPS = 1e-3


def _hubs(copies):
    """`copies` times: hubs of 0 to 40 neighbours of their own, in a shuffled order of ids, with the hubs
    of a copy on a path."""
    lens = np.tile(np.arange(41), copies)
    hubs = lens.size
    src = np.repeat(np.arange(hubs), lens)
    dst = hubs + np.arange(src.size)
    path = np.array([i for i in range(hubs - 1) if i % 41 not in (0, 40)])
    src, dst = np.concatenate([src, path]), np.concatenate([dst, path + 1])
    n = int(hubs + lens.sum())
    relabel = np.random.default_rng(copies).permutation(n)
    return n, relabel[src].astype(np.int32), relabel[dst].astype(np.int32)


def _two_steps(ref, Y, precond):
    """Two steps of (preconditioned) CG from zero in float64."""
    m = 1.0 / (ref["deg"].astype(np.float64) + EPS)[:, None] if precond else 1.0
    x, r = np.zeros_like(Y), Y.copy()
    p = m * r
    rz = np.sum(r * m * r, axis=0)
    for _ in range(2):
        ap = O.laplacian_matvec(ref, EPS, p)
        al = rz / np.sum(p * ap, axis=0)
        x += al * p
        r -= al * ap
        new = np.sum(r * m * r, axis=0)
        p = m * r + new / rz * p
        rz = new
    return x


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("precond", [False, True])
@pytest.mark.parametrize("kc", [4, 12, 20, 32, 48, 100, 128, 132, 256])
def test_resident_rows_of_every_step_length(monkeypatch, kc, precond, weighted):
    """Two steps hold two sweeps of the operator and the true residual a third.  A sweep's rounding is
    at most 42 units of 2^-24 of the sum of its terms' sizes, 2.5e-6, and the steps grow it by the ratio
    of that sum to the result and by r's cancellation, a few each: 1e-4 covers both; a neighbour
    left out, doubled or taken from another row moves a column by its own size."""
    monkeypatch.setenv("ERC_CG_MODE", "resident")
    n, src, dst = _hubs(8)
    w = synth.random_positive(src.size, 6, 0.5, 2.0) if weighted else None
    g, ref = build_both(n, src, dst, w)
    Y = erc.erc_jl_rhs(g, 5, 256, 0, kc)
    fn = erc.erc_batched_pcg_timed if precond else erc.erc_batched_cg_timed
    X, iters, relres, st, _, path = fn(g, EPS, Y, kc, 1e-6, max_iter=2)
    assert path == 1 and st == erc.ERC_ERR_NOT_CONVERGED and np.all(host(iters) == 2)
    X64 = host(X).astype(np.float64)[:, :kc]
    Y64 = host(Y).astype(np.float64)[:, :kc]
    Xr = _two_steps(ref, Y64, precond)
    assert np.all(np.linalg.norm(X64 - Xr, axis=0) <= 1e-4 * np.linalg.norm(Xr, axis=0))
    rest = Y64 - O.laplacian_matvec(ref, EPS, X64)
    true = np.linalg.norm(rest, axis=0) / np.linalg.norm(Y64, axis=0)
    np.testing.assert_allclose(host(relres), true, rtol=1e-4)
