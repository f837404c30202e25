"""Memory that only makes calls faster is done without when it is refused: the
list of nodes with neighbours, and the scratch of split sampling, which never
takes what the call needs after it."""
import threading

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


class Limited:
    """torch's allocator: sizes recorded, request number `at` refused once, and
    nothing beyond `limit` bytes held at a time."""

    def __init__(self, M):
        inner = M.torch_allocator()
        self.mu, self.at, self.limit, self.held = threading.Lock(), -1, None, 0
        self.sizes, self.size = [], {}

        def alloc(nbytes, ctx, stream):
            with self.mu:
                self.sizes.append(nbytes)
                if len(self.sizes) - 1 == self.at or (self.limit is not None and self.held + nbytes > self.limit):
                    return None
                p = inner._keep[0](nbytes, ctx, stream)
                if p:
                    self.size[p] = nbytes
                    self.held += nbytes
                return p

        def free(p, nbytes, ctx, stream):
            with self.mu:
                self.held -= self.size.pop(p)
            inner._keep[1](p, nbytes, ctx, stream)

        kinds = dict(M.Allocator._fields_)
        a, f = kinds["alloc"](alloc), kinds["free"](free)
        self._keep = (a, f, inner)
        self.struct = M.Allocator(a, f, None)


def test_graph_without_the_node_list(M, monkeypatch):
    n, k = 100_000, 5
    i = np.arange(20_000)  # a path; the other nodes have no neighbour
    g = synth.from_edges(n, i, i + 1)
    colors = synth.balanced_colors(n, k, 1)
    want = M.Tables(M.Graph.from_csr(g), colors, k, 64)
    al = Limited(M)
    monkeypatch.setattr(M, "torch_allocator", lambda: al)
    M.Graph.from_csr(g).free()
    lists = [j for j, b in enumerate(al.sizes) if b == 4 * n]
    assert len(lists) == 2  # first hub chunks, then the list
    al.sizes.clear()
    al.at = lists[-1]
    G = M.Graph.from_csr(g)
    al.at = -1
    T = M.Tables(G, colors, k, 64)
    for h in range(1, k + 1):
        assert np.array_equal(T.read(h), want.read(h)) and T.total(h) == want.total(h)


def test_star_samples_beside_split_scratch(M, monkeypatch):
    g, k, n = synth.chung_lu(200_000, 600_000, 2.5, seed=3), 5, 1 << 20
    colors = synth.balanced_colors(g.n, k, 1)
    M.sigma(k)
    want = M.Tables(M.Graph.from_csr(g), colors, k, 64, skip_round=True).estimate(k, 7, n, star_samples=1000)
    al = Limited(M)
    monkeypatch.setattr(M, "torch_allocator", lambda: al)
    T = M.Tables(M.Graph.from_csr(g), colors, k, 64, skip_round=True)
    # room for the split scratch (4 (h + 1) bytes per sample), not for the star index on top of it
    al.limit = al.held + 4 * (k + 1) * n + (2 << 20)
    got = T.estimate(k, 7, n, star_samples=1000)
    al.limit = None
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
