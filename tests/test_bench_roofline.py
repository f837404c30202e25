"""The benchmark's byte models (no GPU): bytes of the first planes that the build
kernels read and write, and the sampler's counted bytes over the time of both
kernels of split sampling."""
import numpy as np
import pytest

import bench
import synth


def test_plane_widths():
    # largest degree 1000, k = 5: (1000 / 5)^(h-1) passes 2^30 at h = 5
    d = np.array([1000] + [3] * 100_000)
    assert bench.plane_widths(d, 5) == ({1: 4, 2: 4, 3: 4, 4: 4, 5: 8}, {1: 4, 2: 4, 3: 4, 4: 8})
    assert set(bench.plane_widths(np.full(100, 4), 8)[0].values()) == {4}
    # no edges, and a clique: the walks, 7! (127 / 8)^7, decide
    assert set(bench.plane_widths(np.zeros(3, int), 4)[0].values()) == {4}
    assert bench.plane_widths(np.full(128, 127), 8)[0][8] == 8


def test_build_bytes_of_planes():
    n, nnz = 1000, 8000
    planes = bench.plane_widths(np.array([1000] + [3] * 100_000), 5)
    csr = 8 * (n + 1) + 4 * nnz + n
    assert bench.algorithmic_bytes("gather_h3", n, nnz, 5, 8, planes) == n * (12 * 4 + 8 * 4) + csr
    assert bench.algorithmic_bytes("gather_h4", n, nnz, 5, 8, planes) == n * (16 * 4 + 4 * 8) + csr
    assert bench.algorithmic_bytes("merge_h5", n, nnz, 5, 8, planes) == \
        n * (4 * (4 + 12 + 16) + 4 * (4 + 6 + 8) + 8 * 4 + 8 * 9)


def test_sampler_bytes_over_both_kernels():
    prof = {"sample": (0.740 * 20, 20), "classify": (0.152 * 20, 20), "gather_h4": (0.24 * 20, 20)}
    counted = {"sample": (1.1, 1, 780_000_000), "sample sectors": (0.0, 0, 2_824_000_000)}
    r = bench.kernel_roofline("sample", prof, counted, 6788.3, "measured", None, None)
    assert r["kernel"] == "sample + classify" and r["avg_launch_ms"] == pytest.approx(0.892)
    assert r["frac"] == pytest.approx(2.824e9 / 0.892e-3 / 6788.3e9, abs=1e-4)
    # one kernel that does both
    r = bench.kernel_roofline("sample", {"sample": (1.08, 1)}, counted, 6788.3, "measured", None, None)
    assert r["kernel"] == "sample" and r["frac"] == pytest.approx(2.824e9 / 1.08e-3 / 6788.3e9, abs=1e-4)
    r = bench.kernel_roofline("gather_h4", prof, counted, 6788.3, "measured", 2.4e8, 1e9)
    assert r["achieved"] == pytest.approx(1000.0) and r["dram_gbs"] == pytest.approx(4166.7)


def test_kernel_sources_hold_the_kernels():
    import os
    csrc = os.path.join(bench.ROOT, "paper_2009_03052_gb300", "csrc")
    for kernel, name in bench.KERNEL_SOURCE.items():
        text = open(os.path.join(csrc, name)).read()
        assert "__global__" in text and f"{kernel}_" in text, (kernel, name)
        assert any(f"{kernel}_{tail}kernel(" in text for tail in ("", "tile_")), (kernel, name)
