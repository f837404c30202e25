"""mc_table_nonzeros equals the non-zero entries of the rows as read, for every
level, planes of 4 and 8 bytes, rows of odd width (padded planes) and wide rows,
on graphs of fewer and of more words than the launch has threads."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    assert torch.cuda.is_available()
    import paper_2009_03052_gb300 as M
    M.build()
    M.load()
    return M


def _clique_beside_path(n):
    # the counts and the planes of K_100: wide rows from level 6 on
    a, b = np.triu_indices(100, 1)
    path = np.arange(100, n - 1)
    return synth.from_edges(n, np.concatenate([a, path]), np.concatenate([b, path + 1]))


@pytest.mark.parametrize("n,k,bits", [(5001, 8, 64), (5001, 8, 128), (1, 4, 64), (70001, 6, 64), (70001, 6, 128)])
def test_nonzeros_of_every_level(M, n, k, bits):
    g = _clique_beside_path(n) if n > 100 else synth.from_edges(n, np.zeros(0, np.int64), np.zeros(0, np.int64))
    T = M.Tables(M.Graph.from_csr(g), synth.balanced_colors(g.n, k, 3), k, bits)
    for which in (0, 1):
        for h in range(1, k + 1 - which):
            assert T.nonzeros(h, which) == int(T.read(h, which).any(axis=2).sum()), (h, which)
