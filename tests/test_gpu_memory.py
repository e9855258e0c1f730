"""Kernels are chosen by the device memory a call can get (needs a CUDA device).
BCS_TEST_MEMORY=k makes the device one of k bytes for the library (on the host
only: what does not fit is refused)."""
import ctypes

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


def test_state_that_does_not_fit(gpu, monkeypatch):
    g = wheel(330_000)
    src = np.arange(0, 330_000, 33001)
    ref = oracle.bc_sources(g, src)
    monkeypatch.setenv("BCS_TEST_MEMORY", str(10**9))
    got = gpu.bc_sources(g.row_ptr, g.col, src)  # another kernel
    assert gpu.last_stats()["n_wide_batches"] == 0
    assert float(np.abs(got - ref).max()) <= 1e-12 * float(np.abs(ref).max())
    monkeypatch.setenv("BCS_TEST_MEMORY", str(10**6))
    with pytest.raises(gpu.BcsError) as e:
        gpu.bc_sources(g.row_ptr, g.col, src)
    assert e.value.code == gpu._lib.BCS_ENOMEM


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
