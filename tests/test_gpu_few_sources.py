"""Source lists that one round of CTAs takes: a call is about as fast as one
source per CTA where that is the sooner route, and keeps the pull and the deep
kernels where they are (needs a CUDA device).  The bound on the time, 1.4 times
one source per CTA, leaves room for the search that finds a graph's depth (at
most a quarter on these) and for the timer."""
import time

import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def layers(count, width, more, seed=2):
    """Layers of `width` vertices, every vertex joined to some of the next."""
    rng = np.random.default_rng(seed)
    e = []
    for l in range(count - 1):
        a = np.arange(width) + l * width
        e.append(np.stack([a, a + width], 1))
        e.append(np.stack([np.repeat(a, more), rng.integers(0, width, width * more) + (l + 1) * width], 1))
    return gg.from_edges(count * width, np.unique(np.concatenate(e), axis=0), "layers%dx%d" % (count, width))


def best(fn):
    fn()
    t = []
    for _ in range(9):
        t0 = time.perf_counter()
        fn()
        t.append(time.perf_counter() - t0)
    return min(t)


@pytest.mark.parametrize("g,k", [(layers(38, 400, 5), 32), (layers(38, 150, 5), 300), (gg.cycle(6000), 1),
                                 (gg.cycle(6000), 32), (gg.path(20000), 30), (gg.grid(100, 100), 1),
                                 (layers(60, 300, 20), 1)],
                         ids=lambda x: getattr(x, "name", str(x)))
def test_no_slower_than_one_source_per_cta(gpu, monkeypatch, g, k):
    src = np.random.default_rng(k).choice(g.n, k, replace=False)
    t = best(lambda: gpu.bc_sources(g.row_ptr, g.col, src))
    ref = oracle.bc_sources(g, src)
    assert float(np.abs(gpu.bc_sources(g.row_ptr, g.col, src) - ref).max()) <= 1e-12 * float(np.abs(ref).max())
    monkeypatch.setenv("BCS_LARGE_PATH", "per_source")
    assert t <= 1.4 * best(lambda: gpu.bc_sources(g.row_ptr, g.col, src))


def test_the_pull_kernel_keeps_hubs(gpu):
    g = gg.chung_lu(20000, 2.3, 5.0, 1)
    src = np.random.default_rng(1).choice(g.n, 32, replace=False)
    got = gpu.bc_sources(g.row_ptr, g.col, src)
    assert gpu.last_stats()["n_wide_batches"] > 0
    ref = oracle.bc_sources(g, src)
    assert float(np.abs(got - ref).max()) <= 1e-12 * float(np.abs(ref).max())
