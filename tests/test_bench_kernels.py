"""bench.py's roofline entry names the kernel that took the time and says what
its bytes are, from fixed call statistics (CPU)."""
import sys

import pytest

from conftest import ROOT

sys.path.insert(0, ROOT)
import bench  # noqa: E402

BASE = {"dag_edges": 2.5e8, "work_sources_entries": 1e9, "work_sources_vertices": 1e8, "ms_bcreach_large": 100.0,
        "ms_bcreach_small": 1.0, "n_large_sources": 640, "n_wide_batches": 0, "n_ms_batches": 0, "n_deep_sources": 0}


@pytest.mark.parametrize("st,kernel,share", [({"n_wide_batches": 10}, "k_bcreach_pull", 64),
                                             ({"n_deep_sources": 640}, "k_bcreach_deep", 1),
                                             ({"n_ms_batches": 20}, "k_bcreach_ms", 32), ({}, "k_bcreach_large", 32)])
def test_kernel_and_basis(monkeypatch, st, kernel, share):
    monkeypatch.setattr(bench, "measured_traffic", lambda kind: {"dram_bytes_per_batch": 3.0e9})
    r = bench.roofline({**BASE, **st}, {"sm_mhz": 2070.0}, {"hbm_gbs": 6000.0}, 152)
    assert r["kernel"].startswith(kernel)
    model = 1e9 * (8.0 / share + 2.0 / 8 + 0.25 * 28.0) + 1e8 * 32.0
    assert r["work"]["model_bytes"] == pytest.approx(model)
    if kernel == "k_bcreach_pull":  # measured bytes where there are any
        assert r["basis"] == "measured DRAM bytes" and r["achieved"] == pytest.approx(3.0e10 / 0.1 / 1e9)
        monkeypatch.setattr(bench, "measured_traffic", lambda kind: None)
        r = bench.roofline({**BASE, **st}, {"sm_mhz": 2070.0}, {"hbm_gbs": 6000.0}, 152)
    assert r["basis"].startswith("model") and r["achieved"] == pytest.approx(model / 0.1 / 1e9)
    assert r["frac"] == pytest.approx(r["achieved"] / 6000.0) and r["traffic"] is None
