"""Totals over node ranges, from the root index's prefix (a scan of one tile, of
tiles added up directly, and of more than 2048 tiles) and from the one-pass
sums per treelet, on paths with node counts around the tile and launch limits:
at k = 2 a node's total is its number of neighbours of the other colour."""
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


def _path(n):
    deg = np.full(n, 2, np.int64)
    deg[0] = deg[-1] = 1
    row_ptr = np.concatenate([[0], np.cumsum(deg)])
    both = np.stack([np.arange(n) - 1, np.arange(n) + 1], 1).reshape(-1)
    return row_ptr, both[1:-1].astype(np.uint32)


@pytest.mark.parametrize("n", [2, 4095, 4096, 4097, 70_001, 2048 * 4096, 2048 * 4096 + 1])
def test_range_totals_on_paths(M, n):
    row_ptr, col = _path(n)
    colors = synth.random_colors(n, 2, 11)
    diff = (colors[1:] != colors[:-1]).astype(np.int64)
    per_node = np.concatenate([[0], diff]) + np.concatenate([diff, [0]])
    prefix = np.concatenate([[0], np.cumsum(per_node)])
    T = M.Tables(M.Graph(row_ptr, col, trusted=True), colors, 2, 64)
    assert T.total(2)[0] == int(prefix[-1])
    rng = np.random.default_rng(n)
    ends = {0, 1, n // 2, n - 1, n} | {min(n, 4096 * int(t)) for t in rng.integers(0, n // 4096 + 1, 4)}
    ends = sorted(ends)
    for lo in ends:
        for hi in ends:
            want = int(prefix[hi] - prefix[lo])
            if lo < hi and want % 2 == 0:  # a range's rooted total must hold both roots of a copy or the call refuses it
                assert T.total(2, -1, (lo, hi))[0] == want
                assert T.total(2, 0, (lo, hi))[0] == want
