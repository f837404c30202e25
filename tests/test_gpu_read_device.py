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


@pytest.mark.parametrize("bits", [64, 128])
@pytest.mark.parametrize("make", [lambda: synth.er_1k(), lambda: synth.star(500), lambda: synth.chung_lu(9000, 40000, 2.4, seed=1)])
def test_host_at_any_address(M, bits, make):
    # small levels are widened on the host, the others on the device
    g, k = make(), 5
    T = M.Tables(M.Graph.from_csr(g), synth.balanced_colors(g.n, k, 3), k, bits)
    for which, h in ((0, 1), (0, 2), (0, 4), (0, 5), (1, 1), (1, 3), (1, 4)):
        want = _device_read(M, T, h, which, 0)
        W, b = T.layout(h, which)
        for off in (0, 8, 1):
            buf = np.full(want.size + 64, 0xA5, np.uint8)
            M._check(M.load().mc_read_table(T.handle, h, which, C.c_void_p(buf.ctypes.data + off), want.size, 0,
                                            M._stream_ptr()))
            assert np.array_equal(buf[off:off + want.size], want), (which, h, off)
            assert (buf[:off] == 0xA5).all() and (buf[off + want.size:] == 0xA5).all()
