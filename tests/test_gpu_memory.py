"""Kernels are chosen by the device memory a call can get (needs a CUDA device).
BCS_TEST_MEMORY=k makes the device one of k bytes for the library (on the host
only: what does not fit is refused)."""
import ctypes
import re

import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def wheel(n):
    e = [(0, i) for i in range(1, n)] + [(i, i % (n - 1) + 1) for i in range(1, n)]
    return gg.from_edges(n, np.array(e), "wheel%d" % n)


def test_a_second_call_gets_what_the_first_got(gpu, monkeypatch):
    """The state of 330,000 vertices, 1.1 GB, has to fit three quarters of what
    there is: 2.4 GB, less the 1.1 if what the pool keeps counted as used."""
    g = wheel(330_000)
    src = np.arange(0, 330_000, 3301)
    ref = oracle.bc_sources(g, src)
    monkeypatch.setenv("BCS_TEST_MEMORY", str(2400 * 10**6))
    for _ in range(2):
        got = gpu.bc_sources(g.row_ptr, g.col, src)
        assert gpu.last_stats()["n_wide_batches"] > 0
        assert float(np.abs(got - ref).max()) <= 1e-12 * float(np.abs(ref).max())


@pytest.mark.parametrize("mbytes", [1000, 700, 550, 380, 1])
def test_state_that_does_not_fit(gpu, monkeypatch, mbytes):
    """The pull kernel with 128, 64 and 32 values to a row, another kernel, an error."""
    g = wheel(330_000)
    src = np.arange(0, 330_000, 3301)
    ref = oracle.bc_sources(g, src)
    monkeypatch.setenv("BCS_TEST_MEMORY", str(mbytes * 10**6))
    if mbytes == 1:
        with pytest.raises(gpu.BcsError) as e:
            gpu.bc_sources(g.row_ptr, g.col, src)
        assert e.value.code == gpu._lib.BCS_ENOMEM
        return
    for fp32, tol in ((False, 1e-12), (True, 1e-5)):
        got = gpu.bc_sources(g.row_ptr, g.col, src, delta_fp32=fp32)
        assert (gpu.last_stats()["n_wide_batches"] > 0) == (mbytes > 400)
        assert float(np.abs(got - ref).max()) <= tol * float(np.abs(ref).max())


def test_narrow_rows_with_reach_and_ident(gpu, monkeypatch, capfd):
    """From the memory for one slab of 256 sources down to none: all widths."""
    monkeypatch.setenv("BCS_LARGE_PATH", "wide_all")
    monkeypatch.setenv("BCS_TRACE", "1")
    g = gg.with_twins_and_pendants(gg.chung_lu(6000, 2.3, 8.0, 1), 1, 900, 1500, 100)
    ref = oracle.bc(g)
    widths = set()
    for kbytes in np.geomspace(4_000, 120_000, 24).astype(int):
        monkeypatch.setenv("BCS_TEST_MEMORY", str(int(kbytes) * 1000))
        for kw, tol in ({}, 1e-12), ({"unequal": True}, 1e-12), ({"delta_fp32": True}, 1e-5):
            try:
                got = gpu.bc_shattered(g.row_ptr, g.col, **kw)
            except gpu.BcsError as e:
                assert e.code == gpu._lib.BCS_ENOMEM
                continue
            assert float(np.abs(got - ref).max()) <= tol * float(np.abs(ref).max())
        widths |= set(re.findall(r"(\d+) values to a row", capfd.readouterr().err))
    assert widths == {"32", "64", "128", "256"}


def test_more_than_two_to_the_24_vertices(gpu, monkeypatch):
    """Two hubs with 8.5 million leaves each, one batch of sources: a leaf of the
    first hub leaves it n - 2 and the other its leaves.  The whole GPU searches,
    with 64 values to a row in 30 GB."""
    half = 8_500_000
    n = 2 * half + 2
    deg = np.ones(n, np.int64)
    deg[:2] = half + 1
    rp = np.concatenate([[0], np.cumsum(deg)])
    leaves = np.arange(2, n, dtype=np.int32)
    col = np.concatenate([np.int32([1]), leaves[:half], np.int32([0]), leaves[half:],
                          np.zeros(half, np.int32), np.ones(half, np.int32)])
    src = np.arange(2, 2 + 64 * 5, 5)
    monkeypatch.setenv("BCS_TEST_MEMORY", str(30 * 10**9))
    got = gpu.bc_sources(rp, col, src)
    assert gpu.last_stats()["n_wide_batches"] > 0
    assert got[0] == 64.0 * (n - 2) and got[1] == 64.0 * half
    assert np.count_nonzero(got) == 2


def test_the_pool_keeps_a_bounded_amount(gpu):
    g = gg.config(1)
    gpu.bc_shattered(g.row_ptr, g.col)
    cuda = ctypes.CDLL("libcuda.so.1")
    dev, pool, keep = ctypes.c_int(), ctypes.c_void_p(), ctypes.c_uint64()
    assert cuda.cuDeviceGet(ctypes.byref(dev), 0) == 0
    assert cuda.cuDeviceGetDefaultMemPool(ctypes.byref(pool), dev) == 0
    release_threshold = 4  # CU_MEMPOOL_ATTR_RELEASE_THRESHOLD
    assert cuda.cuMemPoolGetAttribute(pool, release_threshold, ctypes.byref(keep)) == 0
    assert 0 < keep.value <= 40 * 2**30


def test_a_large_shallow_piece_beside_a_small_deep_one(gpu, monkeypatch):
    """330,000 vertices of two levels take 1.2 GB of the 1.9 there are; with room
    for the 80 levels of a ring of 1,600 in the same batch it would be 2."""
    m = 329_999  # vertices of the rim
    a = np.arange(1600)
    ring = gg.from_edges(1600, np.concatenate([np.stack([a, (a + j) % 1600], 1) for j in range(1, 22)]))
    both = gg.disjoint_union(wheel(m + 1), ring)
    monkeypatch.setenv("BCS_TEST_MEMORY", str(1900 * 10**6))
    got = gpu.bc_shattered_batch(np.array([0, m + 1, both.n]), both.row_ptr, both.col)
    assert gpu.last_stats()["n_wide_batches"] == -(-(m + 1) // 64) + 25
    # of a rim's ordered pairs that are not neighbours the paths cross the hub, those two apart the one between as well
    assert got[0] == m * (m - 3) - m
    assert np.array_equal(got[1:m + 1], np.ones(m))
    ref = oracle.bc(ring)
    assert float(np.abs(got[m + 1:] - ref).max()) <= 1e-12 * float(ref.max())
