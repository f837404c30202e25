"""The merge works on tiles of 8 to 128 nodes and skips nodes without
neighbours when at least an eighth of the nodes have none: every table entry
equals the oracle's at node counts around the tile sizes, with and without
neighbourless nodes, at both count widths and with zero-rooting."""
import numpy as np
import pytest

import synth
from tests.test_gpu_parity import assert_tables_equal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    assert torch.cuda.is_available()
    import paper_2009_03052_gb300 as M
    M.build()
    M.load()
    return M


def _graph(n, alone):
    """About 4n/2 random edges over the first n - alone ids, then shuffled, so
    that the neighbourless nodes lie between the others."""
    rng = np.random.default_rng(n + alone)
    live = max(n - alone, 1)
    e = rng.integers(0, live, size=(2, 4 * live))
    perm = rng.permutation(n)
    return synth.from_edges(n, perm[e[0]], perm[e[1]])


@pytest.mark.parametrize("k,bits,zero_root", [(2, 64, False), (3, 128, False), (5, 64, True), (6, 64, False),
                                              (7, 128, False), (8, 128, True)])
@pytest.mark.parametrize("n,alone", [(1, 1), (9, 0), (130, 13), (130, 40), (1000, 900), (2433, 0)])
def test_tiles_and_neighbourless_nodes(M, oracle, k, bits, zero_root, n, alone):
    g = _graph(n, alone)
    colors = synth.balanced_colors(n, k, 3)
    T = M.Tables(M.Graph.from_csr(g), colors, k, bits, zero_root=zero_root)
    O = oracle.Tables(g, colors, k, bits)
    if not zero_root:
        assert_tables_equal(M, T, O, g, colors, k)
        return
    F = M.Tables(M.Graph.from_csr(g), colors, k, bits)
    assert_tables_equal(M, F, O, g, colors, k)
    for h in range(2, k):
        assert np.array_equal(T.read(h), F.read(h))
    full = F.read(k)
    full[colors != 0] = 0
    assert np.array_equal(T.read(k), full)
