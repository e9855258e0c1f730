"""The shared-memory kernel (a thread per (source, vertex) pair) at the sizes
where it can go wrong: source counts around a CTA's group, rows around four and
32 entries, more levels than its shared memory lists, reach, ident and source
maps, path counts past the 64-bit integers and past the double range; and the
rule that sends shallow pieces of many vertices to the pull kernel (needs a
CUDA device).

Against the oracle; FP64 sums differ from it by the order of additions only
(bar 1e-12 of the largest score), FP32 dependencies by 2^-24 per operation
(bar 1e-5), as in test_gpu_parity.py.
"""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def ladder(layers, width, ring):
    """Complete bipartite layers of `width`, one after the other: width^L paths."""
    e = [(a * width + i, b * width + j) for a, b in zip(range(layers), range(1, layers)) for i in range(width)
         for j in range(width)]
    if ring:
        e += [((layers - 1) * width + i, j) for i in range(width) for j in range(width)]
    return gg.from_edges(layers * width, np.array(e), "ladder%dx%d%s" % (layers, width, "r" if ring else ""))


def check(gpu, g, src=None, fn=None, small=True, **kw):
    ref = oracle.bc(g) if src is None else oracle.bc_sources(g, src)
    scale = max(1.0, float(np.abs(ref).max()))
    for fp32, tol in ((False, 1e-12), (True, 1e-5)):
        if src is None:
            got = (fn or gpu.bc_shattered)(g.row_ptr, g.col, delta_fp32=fp32, **kw)
        else:
            got = gpu.bc_sources(g.row_ptr, g.col, src, delta_fp32=fp32)
        if small:
            assert gpu.last_stats()["n_large_sources"] == 0
        assert float(np.abs(got - ref).max()) <= tol * scale


@pytest.mark.parametrize("g", [gg.path(2), gg.path(3), gg.path(17), gg.cycle(5), gg.cycle(127), gg.cycle(129), gg.cycle(1201),
                               gg.star(32), gg.star(33), gg.star(34), gg.star(70), gg.complete(5), gg.complete(33),
                               gg.complete(34), gg.complete(90), gg.complete_bipartite(3, 37), gg.grid(17, 19),
                               gg.chung_lu(900, 2.3, 8.0, 3)], ids=lambda g: g.name)
def test_small_families(gpu, g):
    check(gpu, g, fn=gpu.bc_plain)
    check(gpu, g, steps=0)


@pytest.mark.parametrize("k", [1, 2, 15, 16, 17, 33, 700])
def test_source_lists(gpu, k):
    """Less than a group, groups with a remainder (and repeats)."""
    for n in (60, 500):
        g = gg.chung_lu(n, 2.5, 6.0, n)
        check(gpu, g, np.random.default_rng(k).integers(0, g.n, k))


def test_reach_ident_and_side_copies(gpu):
    for unequal in (False, True):
        check(gpu, gg.with_twins_and_pendants(gg.grid(12, 20), 3, 60, 90, 20), unequal=unequal)
    check(gpu, gg.config(2, scale_pct=1), side=True)
    check(gpu, gg.disjoint_union(gg.cycle(40), gg.grid(20, 30), gg.path(7), gg.gnp(1, 0.5, 0)), fn=gpu.bc_plain)


@pytest.mark.parametrize("layers,width,ring", [(1100, 2, False), (1100, 2, True), (400, 3, True), (90, 7, True)])
def test_path_counts_past_int64_and_double(gpu, layers, width, ring):
    """2^1099 and 3^200 paths, on the vertices themselves and on classes of
    identical ones (ident = width); the bound on a level's counts passes 2^62
    and 2^900 on the way, the list of levels in shared memory its end."""
    g = ladder(layers, width, ring)
    check(gpu, g, fn=gpu.bc_plain, small=False)
    check(gpu, g)


@pytest.mark.parametrize("graphs,pull", [([gg.chung_lu(1300, 2.5, 8.0, s) for s in range(14)], True),
                                         ([gg.chung_lu(1300, 2.5, 8.0, s) for s in range(3)], False),
                                         ([gg.grid(26, 46)] * 30, False),
                                         ([gg.chung_lu(1300, 2.5, 8.0, s) for s in range(14)] + [gg.grid(26, 46)] * 3
                                          + [gg.cycle(30), gg.chung_lu(300, 2.5, 8.0, 7)], True)],
                         ids=["shallow", "few", "deep", "mixed"])
def test_shallow_pieces_of_many_vertices_go_to_the_pull_kernel(gpu, graphs, pull):
    """Both routes against the oracle, and which one was taken."""
    g = gg.disjoint_union(*graphs)
    check(gpu, g, small=False)
    st = gpu.last_stats()
    assert (st["n_wide_batches"] > 0) == pull
    if not pull:
        assert st["n_large_sources"] == 0


@pytest.mark.parametrize("g", [gg.path(1), gg.path(2), gg.star(40), gg.chung_lu(300, 2.3, 8.0, 2), gg.chung_lu(1300, 2.3, 20.0, 2),
                               gg.star(2300), gg.star(4500), gg.chung_lu(4001, 2.3, 8.0, 2), gg.complete(300), gg.cycle(3001),
                               gg.disjoint_union(gg.grid(60, 50), gg.path(9), gg.gnp(3, 0.0, 0), gg.star(900)),
                               ladder(1100, 2, False), ladder(1900, 2, True)], ids=lambda g: g.name)
def test_without_allocations(gpu, g):
    """The allocation-free call on both sides of the shared memory, hubs taken
    by whole warps (up to eight of a warp's rows, and more), several
    components, path counts past the double range."""
    import torch
    ref = oracle.bc(g)
    scale = max(1.0, float(np.abs(ref).max()))
    rp, col = torch.from_numpy(g.row_ptr).cuda(), torch.from_numpy(g.col).cuda()
    for fp32, tol in ((False, 1e-12), (True, 1e-5), (False, 1e-12)):
        got = gpu.bc_plain_noalloc(rp, col, delta_fp32=fp32).cpu().numpy()
        assert float(np.abs(got - ref).max()) <= tol * scale
