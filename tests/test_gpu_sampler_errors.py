"""A sampler call that reports an error leaves its output arrays as they were."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2609_27209_gb300 import erc, synth

from ._gpu import dev, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("induced", [1, 0])
@pytest.mark.parametrize("kind", [erc.ERC_SAMPLE_NODES, erc.ERC_SAMPLE_EDGES])
@pytest.mark.parametrize("bad", ["above one", "negative", "nan", "all zero", "all below 2^-41"])
def test_failed_sampler_call_writes_no_output(bad, kind, induced):
    _, src, dst, _ = synth.random_connected(20000, 60000, seed=7, weighted=False)
    g = erc.erc_build_laplacian(20000, to_dev(src), to_dev(dst))
    count = g.n if kind == erc.ERC_SAMPLE_NODES else g.m
    p = np.full(count, 1.0 / count, np.float32)
    if bad in ("above one", "negative", "nan"):
        p[count - 3] = {"above one": 1.5, "negative": -1e-3, "nan": np.nan}[bad]
    else:
        p[:] = 0.0 if bad == "all zero" else 2.0 ** -42
    prob = to_dev(p)
    nodes = torch.full((g.n,), -7, dtype=torch.int32, device=dev())
    edges = torch.full((g.m,), -7, dtype=torch.int32, device=dev())
    L = erc.lib()
    size = L.erc_sample_workspace_size(g.n, g.m, 900)
    ws = torch.empty(size, dtype=torch.uint8, device=dev())
    gc, n_s, m_s = g.c(), ctypes.c_int32(-1), ctypes.c_int64(-1)
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    st = L.erc_sample_subgraph(ctypes.byref(gc), kind, ptr(prob), 900, 3, 0, induced, ptr(nodes),
                               ctypes.byref(n_s), ptr(edges), ctypes.byref(m_s), ptr(ws), size,
                               ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == erc.ERC_ERR_INVALID_ARG and n_s.value == 0 and m_s.value == 0
    torch.cuda.synchronize()
    assert bool((nodes == -7).all()) and bool((edges == -7).all())
