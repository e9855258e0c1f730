"""Path counts past the double range that come from ident rather than from the
degrees (needs a CUDA device)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def ring_of_layers(layers, k):
    """Layers of k identical vertices in a ring, neighbouring ones joined
    completely: (row_ptr, col)."""
    n = layers * k
    cols = []
    for l in range(layers):
        near = sorted([(l - 1) % layers, (l + 1) % layers])
        row = np.concatenate([np.arange(m * k, (m + 1) * k, dtype=np.int32) for m in near])
        cols.append(np.tile(row, k))
    return np.arange(n + 1, dtype=np.int64) * (2 * k), np.concatenate(cols)


@pytest.mark.parametrize("path", ["wide_all", "deep_all", None])
def test_merged_ring(gpu, monkeypatch, path):
    """240 layers of 400: merged and split again a ring of 240 vertices of degree
    2 and ident 400, with 400^119 = 2^1028 shortest paths to the far layer.  All
    vertices are alike: bc is the sum of (distance - 1) over the others.  FP64
    sums of 240 terms round to 1e-13 at most, FP32 dependencies to 240 x 2^-24."""
    layers, k = 240, 400
    rp, col = ring_of_layers(layers, k)
    if path:
        monkeypatch.setenv("BCS_LARGE_PATH", path)
    half = layers // 2
    want = 2 * k * sum(j - 1 for j in range(1, half)) + k * (half - 1) + (k - 1)
    for fp32, tol in ((False, 1e-12), (True, 2e-5)):
        got = gpu.bc_shattered(rp, col, resplit=True, delta_fp32=fp32)
        st = gpu.last_stats()
        assert st["n_rounds"] > 0 and st["n_merged"] == layers
        assert (st["n_wide_batches"] > 0) == (path == "wide_all")
        assert float(np.abs(got - want).max()) <= tol * want
