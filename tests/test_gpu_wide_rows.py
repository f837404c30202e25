"""Table rows keep the low 4 or 8 bytes of their counts in a first plane; a
row with a larger count is wide and keeps the upper parts in a second one.
Graphs whose average hides the large counts (so that the narrow plane is
chosen) make wide rows of both kinds: every table entry, the totals and the
samples must still equal the oracle's.

  clique: K_128 with pendant nodes beside a long path, k = 8: counts of level
          7 above 2^32 in the clique (hubs) and sums of level 6 at its
          pendants, in planes of 4 bytes;
  stars:  two joined centres with 16,000 leaves each, k = 8: counts of levels
          7 and 8 above 2^64 at the centres and the leaves, in planes of 8.
"""
import numpy as np
import pytest

import synth
from tests.test_gpu_parity import assert_samples_equal, assert_tables_equal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    assert torch.cuda.is_available()
    import paper_2009_03052_gb300 as M
    M.build()
    M.load()
    return M


def _clique_and_path(n):
    a, b = np.triu_indices(128, 1)
    pend = np.arange(128, 428)
    path = np.arange(428, n - 1)
    return synth.from_edges(n, np.concatenate([a, pend, path]), np.concatenate([b, pend % 128, path + 1]))


def _two_stars(leaves):
    i = np.arange(2, 2 * leaves + 2)
    return synth.from_edges(2 * leaves + 2, np.concatenate([[0], i]), np.concatenate([[1], i % 2]))


@pytest.mark.parametrize("bits", [64, 128])
def test_clique_beside_a_path(M, oracle, bits):
    g, k = _clique_and_path(12000), 8
    colors = synth.balanced_colors(g.n, k, 5)
    T = M.Tables(M.Graph.from_csr(g), colors, k, bits)
    O = oracle.Tables(g, colors, k, bits)
    assert int(T.read(k)[:, :, 0].max()) > 1 << 32
    assert_tables_equal(M, T, O, g, colors, k)
    for h in range(6, k + 1):
        assert T.total(h) == O.total(h)
        assert_samples_equal(T, O, h, 7, 100, 400)


def test_two_stars(M, oracle):
    g, k = _two_stars(16000), 8
    colors = synth.balanced_colors(g.n, k, 6)
    T = M.Tables(M.Graph.from_csr(g), colors, k, 128)
    O = oracle.Tables(g, colors, k, 128)
    assert int(T.read(k - 1)[:, :, 1].max()) > 0  # above 2^64 at level k - 1
    assert_tables_equal(M, T, O, g, colors, k)
    for h in (7, 8):
        assert T.total(h) == O.total(h)
        assert_samples_equal(T, O, h, 9, 0, 300)
