"""The pull kernel (pieces of small BFS depth that do not fit shared memory)
at the sizes where its pieces meet: slabs of 256 sources, units of 16 rows,
rows of 64 entries, rows cut into items, and path counts leaving 32 bits, 64
bits and the range kept without a scale (needs a CUDA device).

Against the oracle; FP64 sums differ from it by the order of additions only
(bar 1e-12 of the largest score), FP32 dependencies by 2^-24 per operation
(bar 1e-5), as in test_gpu_parity.py.
"""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def check(gpu, g, src=None, **kw):
    ref = oracle.bc(g) if src is None else oracle.bc_sources(g, src)
    scale = max(1.0, float(np.abs(ref).max()))
    for fp32, tol in ((False, 1e-12), (True, 1e-5)):
        if src is None:
            got = gpu.bc_shattered(g.row_ptr, g.col, delta_fp32=fp32, **kw)
        else:
            got = gpu.bc_sources(g.row_ptr, g.col, src, delta_fp32=fp32)
        assert gpu.last_stats()["n_wide_batches"] > 0
        assert float(np.abs(got - ref).max()) <= tol * scale


@pytest.fixture(autouse=True)
def every_piece(monkeypatch):
    monkeypatch.setenv("BCS_LARGE_PATH", "wide_all")


def joined(hub_degree, n, seed):
    """A sparse random graph whose vertex 0 has the given degree."""
    rng = np.random.default_rng(seed)
    ring = np.stack([np.arange(n), (np.arange(n) + 1) % n], 1)
    more = rng.integers(0, n, (2 * n, 2))
    hub = np.stack([np.zeros(hub_degree, np.int64), 1 + rng.choice(n - 1, hub_degree, replace=False)], 1)
    e = np.concatenate([ring, more, hub])
    e = np.unique(np.sort(e[e[:, 0] != e[:, 1]], 1), axis=0)
    zero = (e[:, 0] == 0)
    return gg.from_edges(n, np.concatenate([e[~zero], np.sort(hub, 1), [[0, n - 1], [0, 1]]]))


@pytest.mark.parametrize("n", [15, 16, 17, 255, 256, 257, 600])
def test_edges_of_units_and_slabs(gpu, n):
    check(gpu, gg.with_twins_and_pendants(gg.gnp(n, min(1.0, 5.0 / n), n), n, 3, 4, 1))


@pytest.mark.parametrize("k", [1, 31, 32, 33, 64, 65, 255, 256, 257, 513])
def test_source_lists_of_every_remainder(gpu, k):
    g = gg.grid(30, 21)
    src = np.random.default_rng(k).integers(0, g.n, k)  # repeats allowed
    check(gpu, g, src)


@pytest.mark.parametrize("degree", [62, 63, 64, 65, 128, 129, 1000, 4094, 4097, 8300])
def test_rows_around_the_list_and_the_items(gpu, degree):
    """Rows of 64 entries fit a warp's list; longer ones are cut into items of
    64, past 4,096 entries into 64 items of several lists."""
    n = 700 if degree < 600 else 9000
    g = joined(degree, n, degree)
    check(gpu, g, np.concatenate([[0, 1, n - 1], np.random.default_rng(0).choice(n, 300, replace=False)]))


@pytest.mark.parametrize("k,layers", [(30, 12), (400, 10), (2, 60), (60, 115)])
def test_path_counts_past_each_width(gpu, k, layers):
    """Layers of k vertices, consecutive ones joined completely: k^(l-1) paths
    to layer l (30^11 ~ 2^54, 400^9 ~ 2^78, 2^59, 60^114 ~ 2^673)."""
    e = []
    for l in range(layers - 1):
        a, b = np.meshgrid(np.arange(k) + l * k, np.arange(k) + (l + 1) * k)
        e.append(np.stack([a.ravel(), b.ravel()], 1))
    g = gg.from_edges(k * layers, np.concatenate(e))
    check(gpu, g, np.array([0, k - 1, k, (layers // 2) * k, k * layers - 1]))


def test_a_call_over_pieces_of_many_sizes(gpu):
    """Pieces on the pull kernel of every size class at once, with reach and
    ident, in one call."""
    sizes = (20, 90, 400, 1500, 3000)
    g = gg.disjoint_union(*[gg.with_twins_and_pendants(gg.chung_lu(n, 2.3, 6.0, n), n, n // 20, n // 10, 3) for n in sizes])
    check(gpu, g)
    check(gpu, g, unequal=True)
