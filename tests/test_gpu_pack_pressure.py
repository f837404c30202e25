"""Packing under memory pressure: a level's requests before its
synchronisation are refused until memory is freed.  From the second level on
the dense rows of the level before it are still held then, so packing frees
them and goes on; only the first level, and the keys and counts of the last,
have nothing to free."""
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


class Tight:
    """torch's allocator; from request number `at` on everything is refused
    until a block is given back.  `events` lists requests ("a", pointer) and
    releases ("f", pointer)."""

    def __init__(self, M):
        inner = M.torch_allocator()
        self.at, self.calls, self.shut, self.events = -1, 0, False, []

        def alloc(nbytes, ctx, stream):
            self.calls += 1
            if self.calls - 1 == self.at:
                self.shut = True
            if self.shut:
                return None
            p = inner._keep[0](nbytes, ctx, stream)
            self.events.append(("a", p))
            return p

        def free(p, nbytes, ctx, stream):
            self.shut = False
            self.events.append(("f", p))
            inner._keep[1](p, nbytes, ctx, stream)

        kinds = dict(M.Allocator._fields_)
        a, f = kinds["alloc"](alloc), kinds["free"](free)
        self._keep = (a, f, inner)
        self.struct = M.Allocator(a, f, None)


@pytest.mark.parametrize("varlen", [False, True])
def test_refused_until_a_release(M, monkeypatch, varlen):
    g = synth.chung_lu(140000, 420000, 2.4, seed=2)  # every array above the sizes carved from chunks
    k = 4
    colors = synth.balanced_colors(g.n, k, 4)
    G = M.Graph.from_csr(g)
    D = M.Tables(G, colors, k, 64)
    want = {(w, h): D.read(h, w) for w in (0, 1) for h in range(1, k + 1 - w)}
    al = Tight(M)
    monkeypatch.setattr(M, "torch_allocator", lambda: al)
    T = M.Tables(G, colors, k, 64)
    built = al.calls  # requests of the build alone
    T.free()
    al.events.clear()
    al.calls = 0
    T = M.Tables(G, colors, k, 64, succinct=True, varlen=varlen)
    events = list(al.events)
    T.free()
    # the requests of packing, cut where a dense level is given back
    dense = {p for kind, p in events[:built]}
    runs, index = [[]], 0
    for kind, p in events:
        if kind == "a":
            if index >= built:
                runs[-1].append(index)
            index += 1
        elif p in dense:
            runs.append([])
    levels = 2 * (k - 1)
    assert len(runs) == levels + 1
    # a cut run: the keys and counts of one level, then the next level's
    # requests before its synchronisation; the first also has the first level's own
    early = [r[2:] for r in runs[1:levels]]
    head = len(early[0])
    assert head >= 1 and len(runs[0]) >= 2 + 2 * head
    early.insert(0, runs[0][-head:])
    for r in early:
        for at in r:
            al.calls, al.at, al.shut = 0, at, False
            try:
                T = M.Tables(G, colors, k, 64, succinct=True, varlen=varlen)
            finally:
                al.at, al.shut = -1, False
            for (w, h), x in want.items():
                assert np.array_equal(T.read(h, w), x), (at, w, h)
            T.free()
