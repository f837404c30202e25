"""A request is drawn with a warp per sample, a lane per sample for latency or a
lane per sample for throughput, by its size; packed tables have no latency
mode.  All draw the same samples: large requests equal the concatenation of
small ones, which start the warp kernel (its samples are checked against the
oracle elsewhere), for both count widths, a treelet, h < k and packed rows."""
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


def _host(parts):
    return [np.concatenate([p[i].cpu().numpy() for p in parts]) for i in range(4)]


@pytest.mark.parametrize("k,h,bits,unrooted,packed", [(4, 4, 64, -1, False), (5, 5, 64, 1, False), (6, 5, 64, -1, True),
                                                      (6, 6, 128, -1, False), (7, 5, 128, -1, True), (8, 8, 128, 3, False)])
def test_sizes_draw_the_same_samples(M, k, h, bits, unrooted, packed):
    g = synth.chung_lu(4000, 30000, 2.4, max_degree=600.0, seed=k)
    colors = synth.balanced_colors(g.n, k, 2)
    T = M.Tables(M.Graph.from_csr(g), colors, k, bits, succinct=packed)
    total = 60_001
    whole = _host([T.sample(h, 5, 17, total, unrooted=unrooted)])          # throughput
    middle = _host([T.sample(h, 5, 17 + s, min(20_001, total - s), unrooted=unrooted) for s in range(0, total, 20_001)])
    small = _host([T.sample(h, 5, 17 + s, min(1500, 6001 - s), unrooted=unrooted) for s in range(0, 6001, 1500)])
    for a, b, c in zip(whole, middle, small):
        assert np.array_equal(a, b)
        assert np.array_equal(a[:6001], c)
    est = T.estimate(h, seed=5, samples=1500)[1]  # the class histogram of a small request
    cls = T.sample(h, 5, 0, 1500)[3].cpu().numpy()
    assert np.array_equal(est, np.bincount(cls, minlength=len(est)).astype(np.uint64))


def test_wide_rows_below_the_sampled_level(M):
    """Two joined centres with 16,000 leaves each, 128-bit counts, k = 8: rows of
    level 7 are wide, so a large request takes the kernel that reads them in
    line.  The same samples in requests of a warp per sample."""
    i = np.arange(2, 32002)
    g = synth.from_edges(32002, np.concatenate([[0], i]), np.concatenate([[1], i % 2]))
    k = 8
    T = M.Tables(M.Graph.from_csr(g), synth.balanced_colors(g.n, k, 6), k, 128)
    assert int(T.read(k - 1)[:, :, 1].max()) > 0
    count, part = 60000, 4000
    big = [x.cpu().numpy() for x in T.sample(k, 11, 0, count)]
    for lo in range(0, count, part):
        small = T.sample(k, 11, lo, part)
        for a, b in zip(big, small):
            assert np.array_equal(a[lo:lo + part], b.cpu().numpy()), lo
