"""Plain and sampled calls on graphs of many components: a call's time goes with
the vertices its sources reach, not with the graph's square (needs a CUDA
device)."""
import time

import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def copies(g, count):
    e = g.edges()
    return gg.from_edges(count * g.n, (e[None] + (np.arange(count) * g.n)[:, None, None]).reshape(-1, 2))


def best(fn):
    fn()
    t = []
    for _ in range(9):
        t0 = time.perf_counter()
        fn()
        t.append(time.perf_counter() - t0)
    return min(t)


@pytest.mark.parametrize("g,count", [(gg.path(30), 1000), (gg.cycle(9), 5000), (gg.chung_lu(100, 2.3, 6.0, 1), 400)],
                         ids=["paths", "cycles", "chung_lu"])
def test_no_slower_than_one_source_per_cta(gpu, monkeypatch, g, count):
    """1.4 times that: the route's search for the components, and the timer."""
    many = copies(g, count)
    src = np.random.default_rng(2).choice(many.n, 200, replace=False)
    calls = [lambda: gpu.bc_plain(many.row_ptr, many.col), lambda: gpu.bc_sources(many.row_ptr, many.col, src)]
    ref = np.tile(oracle.bc(g), count)
    assert float(np.abs(calls[0]() - ref).max()) <= 1e-12 * max(1.0, float(np.abs(ref).max()))
    ref = oracle.bc_sources(many, src)
    assert float(np.abs(calls[1]() - ref).max()) <= 1e-12 * max(1.0, float(np.abs(ref).max()))
    t = [best(c) for c in calls]
    monkeypatch.setenv("BCS_LARGE_PATH", "per_source")
    for x, c in zip(t, calls):
        assert x <= 1.4 * best(c)


def test_one_large_component_among_small_ones(gpu):
    big = gg.chung_lu(9000, 2.3, 8.0, 3)
    g = gg.disjoint_union(big, copies(gg.cycle(9), 300))
    got = gpu.bc_plain(g.row_ptr, g.col)
    assert gpu.last_stats()["n_wide_batches"] > 0  # the pull kernel keeps it
    ref = oracle.bc(g)
    assert float(np.abs(got - ref).max()) <= 1e-12 * float(np.abs(ref).max())
