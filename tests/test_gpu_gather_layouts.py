"""The neighbour sums pick their lanes per row, units per lane and neighbours at
once by the row's units and the average degree; schedules 4 and 5 fold the
lanes.  Every schedule gives the oracle's tables at every k, on a sparse and a
denser graph with hubs, at both count widths."""
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
    yield M
    M.autotune(1)


@pytest.mark.parametrize("k", [3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("bits", [64, 128])
@pytest.mark.parametrize("m", [1200, 4000])
def test_every_layout(M, oracle, k, bits, m):
    g = synth.chung_lu(601, m, 2.4, max_degree=150.0, seed=k + m)
    colors = synth.balanced_colors(g.n, k, 4)
    G = M.Graph.from_csr(g)
    n, nnz, maxd = G.info()
    M.autotune(0)
    first = None
    for schedule in range(7):
        for h in range(2, k):
            M.autotune_set(0, k, bits, h, n, nnz, maxd, schedule)
        T = M.Tables(G, colors, k, bits)
        if first is None:
            O = oracle.Tables(g, colors, k, bits)
            assert_tables_equal(M, T, O, g, colors, k)
            first = [T.read(h, 1) for h in range(1, k)] + [T.read(k)]
        else:
            for a, b in zip(first, [T.read(h, 1) for h in range(1, k)] + [T.read(k)]):
                assert np.array_equal(a, b), schedule
