"""Tables with wide rows through every sampling mode: requests large enough for
the latency mode, split sampling of less and of more than one wave, and the
one-kernel form without scratch give the samples of small requests (a warp each)
at the same indices; and rebuilding such tables for a colouring with other wide
rows, eagerly and replayed, leaves what a fresh build makes.

  clique: K_128 with pendant nodes beside a path, k = 8: 4-byte planes, counts
          above 2^32, in 64 and 128 bits;
  stars:  two joined centres with leaves, k = 8, 128 bits: 8-byte planes, counts
          above 2^64.
"""
import numpy as np
import pytest

import synth
from tests.test_gpu_wide_rows import _clique_and_path, _two_stars

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    assert torch.cuda.is_available()
    import paper_2009_03052_gb300 as M
    M.build()
    M.load()
    return M


def _tables(M, name, bits, seed=5):
    g = _clique_and_path(12000) if name == "clique" else _two_stars(16000)
    G = M.Graph.from_csr(g)
    return g, G, M.Tables(G, synth.balanced_colors(g.n, 8, seed), 8, bits)


@pytest.mark.parametrize("name,bits", [("clique", 64), ("clique", 128), ("stars", 128)])
def test_every_mode_draws_the_same_samples(M, name, bits):
    _, _, T = _tables(M, name, bits)
    for h in (7, 8):
        for n in (20_000, 60_000, 170_000):
            got = [x.cpu().numpy() for x in T.sample(h, 11, 0, n)]
            for at in (0, n // 2, n - 500):
                want = [x.cpu().numpy() for x in T.sample(h, 11, at, 500)]
                for x, y in zip(got, want):
                    assert np.array_equal(x[at:at + 500], y), (h, n, at)
            hits = np.bincount(got[3], minlength=M.num_classes(h))
            M.sigma(h)
            assert np.array_equal(T.estimate(h, 11, n)[1], hits)
            T.total(h)
            assert np.array_equal(T.estimate_noalloc(h, 11, n)[1], hits)


def _same(A, B):
    for w in (0, 1):
        for h in range(1, 9 - w):
            assert np.array_equal(A.read(h, w), B.read(h, w)), (w, h)
    for h in (6, 7, 8):
        assert A.total(h) == B.total(h)
        for n in (300, 20_000, 60_000):
            for x, y in zip(A.sample(h, 3, 0, n), B.sample(h, 3, 0, n)):
                assert np.array_equal(x.cpu().numpy(), y.cpu().numpy()), (h, n)


@pytest.mark.parametrize("name,bits", [("clique", 64), ("stars", 128)])
@pytest.mark.parametrize("replay", [False, True])
def test_rebuild_with_other_wide_rows(M, name, bits, replay):
    import torch
    g, G, T = _tables(M, name, bits)
    # few colours near the large counts (no wide row), then all of them again
    few = np.zeros(g.n, np.uint8)
    few[::3] = 1
    many = synth.balanced_colors(g.n, 8, 9)
    buf = torch.as_tensor(few).cuda()
    for h in (6, 7):
        T.total(h)
    if replay:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            T.rebuild(buf)
        torch.cuda.current_stream().wait_stream(side)
        T.status()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            T.rebuild(buf)
    for colors in (few, many, few, synth.balanced_colors(g.n, 8, 5)):
        buf.copy_(torch.as_tensor(colors))
        if replay:
            graph.replay()
            torch.cuda.synchronize()
        else:
            T.rebuild(buf)
        T.status()
        F = M.Tables(G, colors, 8, bits)
        if colors is few:
            for w in (0, 1):
                for h in range(1, 9 - w):
                    assert np.array_equal(T.read(h, w), F.read(h, w)), (w, h)
            assert [T.total(h) for h in (6, 7, 8)] == [F.total(h) for h in (6, 7, 8)]
        else:
            _same(T, F)
        F.free()
