"""Calls from several host threads at once, each on its own stream: kernels
whose shared memory differs from launch to launch are launched side by side,
so a limit set for one launch must hold for the others.

  builds:  in-place rebuilds at k = 7 and k = 8, whose merges take 40 to 66 KB
           per block, another size on every level;
  samples: estimates at h = 7 and h = 8 without scratch for split sampling, so
           that one kernel holds the class histogram (3 and 44 KB) beside its
           samples' state.
"""
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
    yield M
    M.autotune(1)


def _run(jobs):
    """Each job (a function of a stream) in a thread of its own."""
    import torch
    errors = []
    gate = threading.Barrier(len(jobs))

    def body(job):
        s = torch.cuda.Stream()
        gate.wait()
        try:
            job(s)
        except Exception as e:  # noqa: BLE001 (reported below)
            errors.append(e)
        s.synchronize()

    threads = [threading.Thread(target=body, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_rebuilds_at_two_sizes(M):
    import torch
    g = synth.chung_lu(20000, 80000, 2.4, seed=3)
    G = M.Graph.from_csr(g)
    M.autotune(0)  # every merge by the first schedule
    made = []
    for k in (7, 8):
        c = M.color(G, k, k)
        made.append((k, c, M.Tables(G, c, k, 128)))
    want = [T.read(k) for k, _, T in made]
    torch.cuda.synchronize()

    def rebuilds(T, c):
        def job(s):
            for _ in range(150):
                T.rebuild(c, stream=s)
            T.status(stream=s)
        return job

    _run([rebuilds(T, c) for _, c, T in made])
    for (k, _, T), w in zip(made, want):
        assert np.array_equal(T.read(k), w)


class NoLarge:
    """torch's allocator, refusing requests above 1 MB while `on`."""

    def __init__(self, M):
        inner = M.torch_allocator()
        self.on = False

        def alloc(nbytes, ctx, stream):
            return None if self.on and nbytes > 1 << 20 else inner._keep[0](nbytes, ctx, stream)

        fn = dict(M.Allocator._fields_)["alloc"](alloc)
        self._keep = (fn, inner)
        self.struct = M.Allocator(fn, inner._keep[1], None)


def test_estimates_at_two_sizes(M, monkeypatch):
    import torch
    al = NoLarge(M)
    monkeypatch.setattr(M, "torch_allocator", lambda: al)
    g = synth.chung_lu(5000, 20000, 2.4, seed=4)
    G = M.Graph.from_csr(g)
    made = []
    for k in (7, 8):
        M.sigma(k)
        made.append((k, M.Tables(G, M.color(G, k, k), k, 128)))
    n = 60000  # more than 256 per SM: a lane per sample
    want = [T.estimate(k, 5, n)[1] for k, T in made]
    torch.cuda.synchronize()
    al.on = True
    got = [[] for _ in range(4)]

    def estimates(i, k, T):
        def job(s):
            for _ in range(200):
                got[i].append(T.estimate(k, 5, n, stream=s)[1])
        return job

    _run([estimates(i, *made[i % 2]) for i in range(4)])
    for w, hits in zip(want * 2, got):
        assert len(hits) == 200 and all(np.array_equal(w, x) for x in hits)
