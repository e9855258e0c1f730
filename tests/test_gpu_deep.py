"""The deep kernel (pieces of many BFS levels and small degree; a thread per
(source, vertex) pair) at the sizes where it can go wrong: source counts around
a CTA's group, rows around four and 32 entries, one-vertex levels, several
components, reach and ident, and path counts past the 64-bit integers and past
the double range (needs a CUDA device).

Against the oracle; FP64 sums differ from it by the order of additions only
(bar 1e-12 of the largest score), FP32 dependencies by 2^-24 per operation
(bar 1e-5), as in test_gpu_parity.py.
"""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def every_piece(monkeypatch):
    monkeypatch.setenv("BCS_LARGE_PATH", "deep_all")


def check(gpu, g, src=None, fn=None, **kw):
    ref = oracle.bc(g) if src is None else oracle.bc_sources(g, src)
    scale = max(1.0, float(np.abs(ref).max()))
    for fp32, tol in ((False, 1e-12), (True, 1e-5)):
        if src is None:
            got = (fn or gpu.bc_shattered)(g.row_ptr, g.col, delta_fp32=fp32, **kw)
        else:
            got = gpu.bc_sources(g.row_ptr, g.col, src, delta_fp32=fp32)
        st = gpu.last_stats()
        assert st["n_wide_batches"] == 0 and st["n_ms_batches"] == 0
        assert float(np.abs(got - ref).max()) <= tol * scale


@pytest.mark.parametrize("g", [gg.path(2), gg.path(3), gg.path(300), gg.cycle(5), gg.cycle(1001), gg.star(40), gg.star(66),
                               gg.grid(33, 31), gg.complete(5), gg.complete(40), gg.complete_bipartite(3, 33),
                               gg.random_tree(400, 2)], ids=lambda g: g.name)
def test_small_families(gpu, g):
    check(gpu, g, fn=gpu.bc_plain)
    check(gpu, g, steps=0)


@pytest.mark.parametrize("k", [1, 2, 455, 456, 457, 2000])
def test_source_lists(gpu, k):
    """Fewer sources than CTAs, one each, and groups of several (with repeats)."""
    g = gg.config(4, scale_pct=1)
    check(gpu, g, np.random.default_rng(k).integers(0, g.n, k))


def test_reach_ident_and_several_components(gpu):
    road = gg.config(4, scale_pct=1)
    check(gpu, gg.with_twins_and_pendants(gg.grid(25, 40), 3, 60, 90, 20))
    check(gpu, gg.with_twins_and_pendants(gg.grid(25, 40), 4, 60, 90, 20), unequal=True)
    check(gpu, gg.disjoint_union(gg.cycle(40), gg.grid(20, 30), gg.path(7), gg.gnp(1, 0.5, 0)), fn=gpu.bc_plain)
    check(gpu, road)


def test_path_counts_past_int64_and_double(gpu):
    """A 700 x 700 grid: C(1398, 699) ~ 2^1392 shortest paths between corners
    (the bound on a level's counts passes 2^900 several times on the way)."""
    g = gg.grid(700, 700)
    check(gpu, g, np.array([0, 699, 350 * 700 + 350, g.n - 1, 0]))


def test_the_plan_takes_it_for_deep_pieces_only(gpu, monkeypatch):
    """Without the variable a road graph's block runs on it, a shallow piece does not."""
    monkeypatch.delenv("BCS_LARGE_PATH")
    g = gg.config(4, scale_pct=1)
    ref = oracle.bc(g)
    got = gpu.bc_shattered(g.row_ptr, g.col)
    assert float(np.abs(got - ref).max()) <= 1e-12 * float(np.abs(ref).max())
    st = gpu.last_stats()
    assert st["n_large_sources"] > 10000 and st["n_wide_batches"] == 0 and st["n_ms_batches"] == 0
    g = gg.chung_lu(6000, 2.3, 8.0, 1)
    gpu.bc_shattered(g.row_ptr, g.col)
    assert gpu.last_stats()["n_wide_batches"] > 0
