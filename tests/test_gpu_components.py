"""Connected components on graphs whose first neighbours form long chains (needs
a CUDA device): the labels feed every shattered call, so the check is its
result, and the time of the stage."""
import numpy as np
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [None, 3])
def test_a_long_path(gpu, seed):
    """Numbered along the path every vertex points at the one before: walking
    that chain takes a dependent load per vertex (0.3 us at least: 90 ms for
    300,000), jumping along it some twenty."""
    n = 300_000
    g = gg.path(n) if seed is None else gg.relabel(gg.path(n), seed)
    want = np.sort(2.0 * np.arange(n) * (n - 1 - np.arange(n)))
    ms = []
    for _ in range(3):
        got = gpu.bc_shattered(g.row_ptr, g.col, steps=gpu.STEP_D)
        ms.append(gpu.last_stats()["ms_cc"])
        assert np.array_equal(np.sort(got), want)
    assert min(ms) < 10.0


def test_a_path_of_more_vertices_than_threads(gpu):
    """As above where a kernel's grid of a fixed size has several vertices to a
    thread (walking: 164 ms)."""
    n = 2_000_000
    g = gg.path(n)
    ms = []
    for _ in range(2):
        got = gpu.bc_shattered(g.row_ptr, g.col, steps=gpu.STEP_D)
        ms.append(gpu.last_stats()["ms_cc"])
    assert np.array_equal(got, 2.0 * np.arange(n) * (n - 1 - np.arange(n)))
    assert min(ms) < 10.0


def test_rows_of_a_dense_graph(gpu):
    """200 vertices, all joined: the pieces' rows are written with a thread to a
    row, in less than twice the time of the merging stage (1.4; 2.4 with a warp to
    a row, its 32 rows one after the other)."""
    g = gg.complete(200)
    blocks, ident = [], []
    for _ in range(12):
        got = gpu.bc_shattered(g.row_ptr, g.col, steps=gpu.STEP_D)
        st = gpu.last_stats()
        blocks.append(st["ms_blocks"])
        ident.append(st["ms_ident"])
        assert np.array_equal(got, np.zeros(200))
    assert min(blocks) <= 2.0 * min(ident)
