"""What the autotuner times and picks (needs a CUDA device).  Its choices are
kept per process, so each test has one of its own."""
import os
import re
import subprocess
import sys

import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu


def run(code, **env):
    head = "import numpy as np, graphgen as gg, oracle, paper_1209_6007_gb300 as bcs\n"
    r = subprocess.run([sys.executable, "-c", head + code], cwd=ROOT, env={**os.environ, **env}, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return r.stdout, r.stderr


def test_the_fixed_rule_is_among_the_thresholds(gpu):
    """Pieces of some 900 vertices in numbers: without the autotuner the rule for
    shallow pieces sends them to the pull kernel."""
    out, err = run('''
g = gg.disjoint_union(*[gg.chung_lu(1000, 2.3, 8.0, i) for i in range(48)])
ref = bcs.bc_shattered(g.row_ptr, g.col)
assert bcs.last_stats()["n_wide_batches"] > 0
for _ in range(2):
    got = bcs.bc_shattered(g.row_ptr, g.col, autotune=True)
    assert np.abs(got - ref).max() <= 1e-12 * ref.max()
    assert bcs.last_stats()["small_limit"] in (100 * 1024, 64 * 1024, 40 * 1024)
''', BCS_TRACE="1")
    assert "0" in re.findall(r"tune small/large threshold (\d+) B", err)


def test_a_choice_is_not_taken_where_it_is_not_open(gpu):
    """A grid of 62 x 62, and one with a vertex of 70 more entries: the same size,
    mean degree and depth, but the deep kernel takes rows of up to 64."""
    run('''
a = gg.grid(62, 62)
hub = a.n // 2
b = gg.from_edges(a.n + 70, np.concatenate([a.edges(), np.stack([np.full(70, hub), np.arange(a.n, a.n + 70)], 1)]))
for fp32 in (False, True):
    for g in (a, b, a):
        ref = oracle.bc(g)
        got = bcs.bc_plain(g.row_ptr, g.col, autotune=True, delta_fp32=fp32)
        assert np.abs(got - ref).max() <= (1e-5 if fp32 else 1e-12) * ref.max()
        st = bcs.last_stats()
        # the kernel it says is the one that ran
        assert (st["tuned"] & 2 != 0) == (st["n_wide_batches"] > 0)
        assert (st["tuned"] & 32 != 0) == (st["n_deep_sources"] > 0)
        assert st["tuned"] & (2 | 4 | 8 | 32)
        if g is a: assert st["n_deep_sources"] > 0  # by far the fastest here: so the choice is kept
''')
