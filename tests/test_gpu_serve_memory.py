"""What served requests take from the tables' allocator stays within the
server's memory budget, however many are small and run at once."""
import threading
import time

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


class Counting:
    """torch's allocator with the bytes held and their peak; slow while
    `slow`, so that requests overlap."""

    def __init__(self, M):
        inner = M.torch_allocator()
        self.mu, self.size, self.held, self.peak, self.slow = threading.Lock(), {}, 0, 0, False

        def alloc(nbytes, ctx, stream):
            p = inner._keep[0](nbytes, ctx, stream)
            if p:
                with self.mu:
                    self.size[p] = nbytes
                    self.held += nbytes
                    self.peak = max(self.peak, self.held)
            if self.slow:
                time.sleep(0.01)
            return p

        def free(p, nbytes, ctx, stream):
            with self.mu:
                self.held -= self.size.pop(p)
            inner._keep[1](p, nbytes, ctx, stream)

        kinds = dict(M.Allocator._fields_)
        a, f = kinds["alloc"](alloc), kinds["free"](free)
        self._keep = (a, f, inner)
        self.struct = M.Allocator(a, f, None)


@pytest.mark.parametrize("kind,h,n,budget", [
    ("sample", 5, 64, 2 << 20),
    ("sample", 4, 64, 3 << 20),       # the first request makes the level's root index
    ("estimate", 5, 3000, 3 << 20),
    ("ags", 5, 30000, 8 << 20),
])
def test_small_requests_stay_in_the_budget(M, monkeypatch, kind, h, n, budget):
    al = Counting(M)
    monkeypatch.setattr(M, "torch_allocator", lambda: al)
    g = synth.chung_lu(3000, 12000, 2.4, seed=1)
    G = M.Graph.from_csr(g)
    T = M.Tables(G, synth.balanced_colors(g.n, 5, 2), 5, 64)
    M.sigma(h)
    S = M.Server([T], slots=8, memory_budget=budget)
    al.peak = base = al.held
    al.slow = True
    submit = {"sample": lambda i: S.submit_sample(0, h, 7 + i, n),
              "estimate": lambda i: S.submit_estimate(0, h, 7 + i, n),
              "ags": lambda i: S.submit_estimate(0, h, 7 + i, n, mode=M.MC_EST_AGS, cbar=50, batch=2000)}[kind]
    res = [S.wait(i) for i in [submit(i) for i in range(24)]]
    al.slow = False
    S.free()
    assert al.peak - base <= budget, al.peak - base
    if kind == "sample":
        for i in (0, 23):
            nodes = T.sample(h, 7 + i, 0, n)[0]
            assert np.array_equal(res[i]["nodes"], nodes.cpu().numpy().astype(np.uint32))
