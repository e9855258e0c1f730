"""With FP32 dependencies the bc sums stay FP64 (needs a CUDA device): on graphs
whose dependencies are integers below 2^24, exact in FP32, and whose terms and
sums are integers past 2^24 and below 2^53, the result is exact."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def test_sums_of_many_sources(gpu):
    """251 leaves of a star: each leaves the centre n - 2."""
    n = 100_003
    g = gg.star(n)
    src = 1 + np.random.default_rng(0).choice(n - 1, 251, replace=False)
    got = gpu.bc_sources(g.row_ptr, g.col, src, delta_fp32=True)
    assert gpu.last_stats()["n_wide_batches"] > 0
    centre = int(np.argmax(np.diff(g.row_ptr)))
    assert got[centre] == 251.0 * (n - 2)
    assert np.count_nonzero(got) == 1


@pytest.mark.parametrize("path", [None, "wide_all", "deep_all", "per_source", "batched"])
def test_weighted_terms(gpu, monkeypatch, path):
    """A ring of five with thousands of pendants each: a term is the product of a
    reach and a dependency, some 3,000 x 6,000."""
    if path:
        monkeypatch.setenv("BCS_LARGE_PATH", path)
    pend = [3001, 3011, 3019, 3023, 3037]
    e = [(i, (i + 1) % 5) for i in range(5)]
    n = 5
    for i, p in enumerate(pend):
        e += [(i, n + j) for j in range(p)]
        n += p
    g = gg.from_edges(n, np.array(e))
    got = gpu.bc_shattered(g.row_ptr, g.col, delta_fp32=True)
    assert np.array_equal(got, oracle.bc(g))
