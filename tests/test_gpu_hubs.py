"""Long rows in the steps before Bc-Reach (a warp, a CTA or the GPU takes them
together): components, spanning forest, blocks, copies' rows and BFS orders of
graphs with hubs around the limits of 32, 64, 256 and 2,048 entries, hubs that
are cut vertices of many blocks among them (needs a CUDA device).

Against the oracle; FP64 sums differ from it by the order of additions only
(bar 1e-12 of the largest score), as in test_gpu_parity.py.
"""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def windmill(k, size):
    """A hub that is in k cliques of `size` further vertices each."""
    e = [(0, 1 + c * size + i) for c in range(k) for i in range(size)]
    e += [(1 + c * size + i, 1 + c * size + j) for c in range(k) for i in range(size) for j in range(i)]
    return gg.from_edges(1 + k * size, np.array(e), "windmill%dx%d" % (k, size))


def wheel(n):
    e = [(0, i) for i in range(1, n)] + [(i, i % (n - 1) + 1) for i in range(1, n)]
    return gg.from_edges(n, np.array(e), "wheel%d" % n)


def hubs(n, k, seed):
    """A path with k hubs on it, each next to a random half of the vertices."""
    rng = np.random.default_rng(seed)
    e = [(i, i + 1) for i in range(n - 1)]
    for h in rng.choice(n, k, replace=False):
        for v in rng.choice(n, n // 2, replace=False):
            if abs(int(h) - int(v)) > 1:
                e.append((min(int(h), int(v)), max(int(h), int(v))))
    return gg.from_edges(n, np.unique(np.array(e), axis=0), "hubs%dx%d" % (n, k))


GRAPHS = [windmill(16, 2), windmill(17, 2), windmill(70, 3), windmill(700, 3), windmill(33, 1), wheel(33), wheel(34),
          wheel(66), wheel(2049), wheel(2050), hubs(70, 2, 1), hubs(600, 5, 2), hubs(4200, 3, 3),
          gg.disjoint_union(windmill(90, 4), wheel(300), gg.path(9), hubs(200, 9, 4), gg.complete(40))]


@pytest.mark.parametrize("path", [None, "wide_all"])
@pytest.mark.parametrize("seed", [None, 11])
@pytest.mark.parametrize("g", GRAPHS, ids=lambda g: g.name)
def test_hubs(gpu, monkeypatch, g, seed, path):
    if path:
        monkeypatch.setenv("BCS_LARGE_PATH", path)
    if seed is not None:
        g = gg.relabel(g, seed)
    ref = oracle.bc(g)
    scale = max(1.0, float(np.abs(ref).max()))
    for fn in (gpu.bc_shattered, gpu.bc_plain):
        assert float(np.abs(fn(g.row_ptr, g.col) - ref).max()) <= 1e-12 * scale


@pytest.mark.parametrize("g", [wheel(40000), windmill(13000, 3), gg.complete_bipartite(3, 40000),
                               gg.disjoint_union(wheel(36000), windmill(20, 30), gg.gnp(40, 0.0, 0))], ids=lambda g: g.name)
def test_large_hubs_from_sources(gpu, g):
    """Levels too wide for one CTA: the whole GPU searches."""
    src = np.array([0, 1, g.n - 1, g.n // 2, 17])
    ref = oracle.bc_sources(g, src)
    got = gpu.bc_sources(g.row_ptr, g.col, src)
    assert float(np.abs(got - ref).max()) <= 1e-12 * max(1.0, float(np.abs(ref).max()))
