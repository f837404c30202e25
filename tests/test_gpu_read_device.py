"""mc_read_table into device memory: at any address -- a dst that is not
aligned to a count is filled by copies -- for dense and packed tables, with
and without scratch, every level equals the host read; the bytes around dst
stay as they were."""
import ctypes as C

import numpy as np
import pytest

import synth
from tests.test_gpu_memory_limits import Refusing

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    assert torch.cuda.is_available()
    import paper_2009_03052_gb300 as M
    M.build()
    M.load()
    return M


def _device_read(M, T, h, which, off):
    import torch
    W, b = T.layout(h, which)
    size = T.graph.n * W * b
    buf = torch.full((size + 64,), 0xA5, dtype=torch.uint8, device="cuda")
    assert buf.data_ptr() % 16 == 0
    M._check(M.load().mc_read_table(T.handle, h, which, C.c_void_p(buf.data_ptr() + off), size, 1, M._stream_ptr()))
    x = buf.cpu().numpy()
    assert (x[:off] == 0xA5).all() and (x[off + size:] == 0xA5).all()
    return x[off:off + size]


@pytest.mark.parametrize("bits,kw", [(64, {}), (128, {}), (64, {"succinct": True}), (128, {"varlen": True})])
def test_any_address(M, monkeypatch, bits, kw):
    # K_100 beside a path, k = 8: planes of 4 and 8 bytes, wide rows in both widths
    a, b = np.triu_indices(100, 1)
    path = np.arange(100, 1999)
    g = synth.from_edges(2000, np.concatenate([a, path]), np.concatenate([b, path + 1]))
    k = 8
    al = Refusing(M)
    monkeypatch.setattr(M, "torch_allocator", lambda: al)
    T = M.Tables(M.Graph.from_csr(g), synth.balanced_colors(g.n, k, 3), k, bits, **kw)
    for which, h in ((0, 1), (0, 3), (0, 7), (0, 8), (1, 1), (1, 5), (1, 7)):
        want = T.read(h, which).view(np.uint8).ravel()
        for off in (0, 16, 8, 4, 1):
            assert np.array_equal(_device_read(M, T, h, which, off), want), (which, h, off)
        if kw:
            continue
        al.closed = True  # no scratch
        try:
            for off in (0, 8, 1):
                assert np.array_equal(_device_read(M, T, h, which, off), want), (which, h, off)
        finally:
            al.closed = False
