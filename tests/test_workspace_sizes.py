"""The sampler's workspace covers what a call on it uses, for every graph up to the sizes it was
reported for.  No compute call is made here, so these tests run without a GPU."""
import itertools

import pytest

from paper_2609_27209_gb300 import erc

NODES, EDGES = erc.ERC_SAMPLE_NODES, erc.ERC_SAMPLE_EDGES
# both sides of the entry count where a scan tile grows from 2,048 to 8,192 entries, of the node
# counts where a copy of the marks is dropped, and sizes between
SIZES = [1, 2047, 2049, 169343, 500000, 700000, 900000, (1 << 20) - 1, 1 << 20, (1 << 20) + 1,
         1200000, 2000000, 3000000, 4194304, 4200000, 33000000, 34000000, 100000000]


@pytest.fixture(scope="module")
def size():
    import __graft_entry__

    __graft_entry__.build()
    return erc.lib().erc_sample_workspace_size


def _tiles(count):
    tile = 2048 if count < 1 << 20 else 8192
    return -(-count // tile)


def _used(n, m, kind):
    """Bytes of the arrays one call works on: the weights' prefix sums and every 64th of them, the
    node marks' copies and bits, the edge marks, and a look-back word for each tile of the scan
    over the drawn kind and of the compactions over nodes and edges."""
    count = n if kind == NODES else m
    copies = min(16, max(1, (64 << 20) // n))
    return (8 * count + 8 * (count // 64) + n * copies + n // 8 + m +
            8 * (_tiles(count) + _tiles(n) + _tiles(m)))


@pytest.mark.parametrize("kind", [NODES, EDGES])
def test_sampler_workspace_holds_every_array(size, kind):
    for n, m in itertools.product(SIZES, SIZES):
        assert size(n, m, 100) >= _used(n, m, kind), (n, m)


def test_sampler_workspace_of_a_larger_graph_serves_a_smaller_one(size):
    for m in SIZES:
        sizes = [size(n, m, 100) for n in SIZES]
        assert sizes == sorted(sizes), m
    for n in SIZES:
        sizes = [size(n, m, 100) for m in SIZES]
        assert sizes == sorted(sizes), n


# both sides of the key count (2^21) where the build's sort takes larger tiles, and sizes between
INPUTS = [0, 1, 2047, 2049, 500000, (2 << 20) - 4096, (2 << 20) - 1, 2 << 20, (2 << 20) + 1,
          (2 << 20) + 9000, 2200000, 4194304, 50000000]


@pytest.mark.parametrize("call", ["build", "run", "run_host"])
def test_build_workspace_of_a_larger_graph_serves_a_smaller_one(size, call):
    L = erc.lib()
    f = {"build": L.erc_build_laplacian_workspace_size,
         "run": lambda n, m: L.erc_run_workspace_size(n, m, 64),
         "run_host": lambda n, m: L.erc_run_host_workspace_size(n, m, 64, 256)}[call]
    for m in INPUTS:
        sizes = [f(n, m) for n in SIZES]
        assert sizes == sorted(sizes), m
    for n in SIZES:
        sizes = [f(n, m) for m in INPUTS]
        assert sizes == sorted(sizes), n
