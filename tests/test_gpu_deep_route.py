"""Which calls the deep kernel takes, and its exponents with several sources to a
CTA (needs a CUDA device).

Bars as in test_gpu_deep.py: 1e-12 of the largest score with FP64 dependencies,
1e-5 with FP32."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def check(gpu, got, ref, fp32):
    assert float(np.abs(got - ref).max()) <= (1e-5 if fp32 else 1e-12) * float(np.abs(ref).max())


@pytest.mark.parametrize("g", [gg.path(300), gg.cycle(1001), gg.grid(33, 31), gg.complete(40), gg.star(40),
                               gg.random_tree(400, 2)], ids=lambda g: g.name)
def test_forced(gpu, monkeypatch, g):
    monkeypatch.setenv("BCS_LARGE_PATH", "deep_all")
    gpu.bc_plain(g.row_ptr, g.col)
    assert gpu.last_stats()["n_deep_sources"] == g.n
    src = np.arange(0, g.n, 3)
    gpu.bc_sources(g.row_ptr, g.col, src)
    assert gpu.last_stats()["n_deep_sources"] == src.size


def test_long_rows_are_not_its(gpu, monkeypatch):
    """A row is one thread's work: at most 64 entries."""
    monkeypatch.setenv("BCS_LARGE_PATH", "deep_all")
    for n, takes in ((65, True), (66, False)):
        g = gg.star(n)
        check(gpu, gpu.bc_plain(g.row_ptr, g.col), oracle.bc(g), False)
        assert gpu.last_stats()["n_deep_sources"] == (n if takes else 0)


def test_planned(gpu):
    g = gg.config(4, scale_pct=1)
    gpu.bc_shattered(g.row_ptr, g.col)
    assert gpu.last_stats()["n_deep_sources"] > 10000
    g = gg.chung_lu(6000, 2.3, 8.0, 1)
    gpu.bc_shattered(g.row_ptr, g.col)
    assert gpu.last_stats()["n_deep_sources"] == 0


def ladder(layers, width, cross):
    """Layers of `width`; a vertex joined to all of the next layer (2 of it if not cross)."""
    e = []
    for l in range(layers - 1):
        a = np.arange(width)
        if cross:
            x, y = np.meshgrid(a + l * width, a + (l + 1) * width)
            e.append(np.stack([x.ravel(), y.ravel()], 1))
        else:
            for d in (0, 1):
                e.append(np.stack([a + l * width, (a + d) % width + (l + 1) * width], 1))
    return gg.from_edges(layers * width, np.concatenate(e))


@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("layers,width,cross", [(1100, 2, True), (1250, 3, False)])
def test_several_sources_past_the_double_range(gpu, monkeypatch, fp32, layers, width, cross):
    """2^(l - 1) paths to layer l from one side, and from sources in the middle to
    both: exponents differ between the sources of a CTA."""
    monkeypatch.setenv("BCS_LARGE_PATH", "deep_all")
    g = ladder(layers, width, cross)
    ref = oracle.bc(g)
    check(gpu, gpu.bc_plain(g.row_ptr, g.col, delta_fp32=fp32), ref, fp32)
    assert gpu.last_stats()["n_deep_sources"] == g.n  # 5 to 9 of them on each of 456 CTAs
    check(gpu, gpu.bc_shattered(g.row_ptr, g.col, delta_fp32=fp32, steps=0), ref, fp32)
    assert gpu.last_stats()["n_deep_sources"] == g.n


@pytest.mark.parametrize("fp32", [False, True])
def test_several_sources_with_reach_and_ident_past_the_double_range(gpu, monkeypatch, fp32):
    """The merged layers of a ring: reach and ident of 3, 3^l paths; pendants on
    some of the vertices keep the classes of a layer apart."""
    monkeypatch.setenv("BCS_LARGE_PATH", "deep_all")
    layers, width = 1400, 4
    rng = np.random.default_rng(5)
    e = []
    for l in range(layers):
        x, y = np.meshgrid(np.arange(width) + l * width, np.arange(width) + (l + 1) % layers * width)
        e.append(np.stack([x.ravel(), y.ravel()], 1))
    n = layers * width
    pend = rng.choice(n, n // 8, replace=False)
    g = gg.from_edges(n + pend.size, np.concatenate(e + [np.stack([pend, np.arange(n, n + pend.size)], 1)]))
    ref = oracle.bc(g)
    check(gpu, gpu.bc_shattered(g.row_ptr, g.col, delta_fp32=fp32), ref, fp32)
    st = gpu.last_stats()
    assert layers < st["n_deep_sources"] < n  # merged, several to a CTA
