"""Requests on either side of the sizes where sampling and classification split
into two kernels (h <= 6: four waves of lanes, h >= 7: past the latency mode),
and in the latency mode, give the samples and hits of small requests at the same indices, from dense and
packed tables."""
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


@pytest.mark.parametrize("k,bits,kw", [(4, 64, {}), (6, 128, {}), (6, 64, {"varlen": True}), (7, 128, {}), (7, 128, {"succinct": True})])
def test_both_sides_of_the_split(M, k, bits, kw):
    import torch
    waves = torch.cuda.get_device_properties(0).multi_processor_count * 4 * 1536
    g = synth.chung_lu(20000, 60000, 2.5, seed=k)
    G = M.Graph.from_csr(g)
    T = M.Tables(G, M.color(G, k, 2), k, bits, **kw)
    M.sigma(k)
    for n in (20_000, 50_000, waves - 1, waves, waves + 77):
        got = [x.cpu().numpy() for x in T.sample(k, 21, 5, n)]
        for at in (0, n - 400):
            for x, y in zip(got, T.sample(k, 21, 5 + at, 400)):
                assert np.array_equal(x[at:at + 400], y.cpu().numpy()), (n, at)
        hits = np.bincount(got[3], minlength=M.num_classes(k))
        assert np.array_equal(T.estimate(k, 21, n, first_index=5)[1], hits)
