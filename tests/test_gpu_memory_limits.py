"""Calls at the edge of device memory, with an allocator that refuses: a dense
level still reaches the host when there is no scratch to expand it in, and
packing goes on when a level's arrays do not fit beside the dense rows of the
level before it (whose fill is still queued).
"""
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


class Refusing:
    """torch's allocator, refusing every request while `closed`, and request
    number `at` once."""

    def __init__(self, M):
        inner = M.torch_allocator()
        self.closed, self.at, self.calls = False, -1, 0

        def alloc(nbytes, ctx, stream):
            self.calls += 1
            return None if self.closed or self.calls - 1 == self.at else inner._keep[0](nbytes, ctx, stream)

        fn = dict(M.Allocator._fields_)["alloc"](alloc)
        self._keep = (fn, inner)
        self.struct = M.Allocator(fn, inner._keep[1], None)


@pytest.mark.parametrize("bits", [64, 128])
def test_read_without_scratch(M, monkeypatch, bits):
    # K_100 beside a path, k = 8: planes of 4 and 8 bytes, wide rows in both widths
    a, b = np.triu_indices(100, 1)
    path = np.arange(100, 5000)
    g = synth.from_edges(5001, np.concatenate([a, path]), np.concatenate([b, path + 1]))
    k = 8
    al = Refusing(M)
    monkeypatch.setattr(M, "torch_allocator", lambda: al)
    T = M.Tables(M.Graph.from_csr(g), synth.balanced_colors(g.n, k, 3), k, bits)
    for which, levels in ((0, range(1, k + 1)), (1, range(1, k))):
        for h in levels:
            want = T.read(h, which)
            al.closed = True
            try:
                got = T.read(h, which)
            finally:
                al.closed = False
            assert np.array_equal(got, want), (which, h)


def test_packing_with_one_refusal(M, monkeypatch):
    g = synth.chung_lu(12000, 60000, 2.4, seed=2)
    k = 5
    colors = synth.balanced_colors(g.n, k, 4)
    al = Refusing(M)
    G = M.Graph.from_csr(g)
    want = [M.Tables(G, colors, k, 64).read(h, 0) for h in range(1, k + 1)]
    monkeypatch.setattr(M, "torch_allocator", lambda: al)
    al.calls = 0
    M.Tables(G, colors, k, 64)
    dense = al.calls  # requests of the build alone
    al.calls = 0
    M.Tables(G, colors, k, 64, varlen=True)
    survived = 0
    for at in range(dense, al.calls):
        al.calls, al.at = 0, at
        try:
            T = M.Tables(G, colors, k, 64, varlen=True)
        except M.MotifError as e:
            assert e.status == M.MC_E_NOMEM
            continue
        finally:
            al.at = -1
        survived += 1
        for h in range(1, k + 1):
            assert np.array_equal(T.read(h, 0), want[h - 1]), (at, h)
    assert survived >= 6  # the offset arrays of every level
