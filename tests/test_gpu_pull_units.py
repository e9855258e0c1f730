"""The pull kernel where a wave has few units: the rows of a unit go to several
warps (needs a CUDA device).

Results against the oracle (bars as in test_gpu_pull.py); times against one
source per CTA, the route of these pieces without the pull kernel.
"""
import time

import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def ring(n, k):
    """Every vertex joined to k neighbours on either side."""
    a = np.arange(n)
    return gg.from_edges(n, np.concatenate([np.stack([a, (a + j) % n], 1) for j in range(1, k + 1)]), "ring%dx%d" % (n, k))


@pytest.mark.parametrize("k", [100, 1024, 2048, 4000, 6007])
def test_units_of_every_size(gpu, monkeypatch, k):
    """Slabs of 6,007 rows: units of 1, 2, 4, 8 and 8 rows on 152 SMs."""
    monkeypatch.setenv("BCS_LARGE_PATH", "wide")
    g = gg.chung_lu(6007, 2.3, 9.0, 2)
    src = np.random.default_rng(k).choice(g.n, k, replace=False)
    ref = oracle.bc_sources(g, src)
    for fp32, tol in ((False, 1e-12), (True, 1e-5)):
        got = gpu.bc_sources(g.row_ptr, g.col, src, delta_fp32=fp32)
        assert gpu.last_stats()["n_wide_batches"] > 0
        assert float(np.abs(got - ref).max()) <= tol * float(np.abs(ref).max())


def best(fn):
    fn()
    t = []
    for _ in range(9):
        t0 = time.perf_counter()
        fn()
        t.append(time.perf_counter() - t0)
    return min(t)


@pytest.mark.parametrize("g", [ring(1600, 21), ring(3200, 40)], ids=lambda g: g.name)
def test_no_slower_than_one_source_per_cta(gpu, monkeypatch, g):
    pull = best(lambda: gpu.bc_plain(g.row_ptr, g.col))
    assert gpu.last_stats()["n_wide_batches"] > 0
    monkeypatch.setenv("BCS_LARGE_PATH", "per_source")
    assert pull <= 1.25 * best(lambda: gpu.bc_plain(g.row_ptr, g.col))
