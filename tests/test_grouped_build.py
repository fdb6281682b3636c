"""Graphs built by the partition passes (2^20 edges or more, at most 2^24 vertices) against the oracle:
one edge short of the bound and at it, tile remainders, vertex counts around a bucket's size, all edges
at one vertex, empty rows at the ends, every creation flag and input form, and bad input in the last
edge."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from tests.gpu_util import graph_handle, run

pytestmark = pytest.mark.gpu
M0 = 1 << 20


def _rand(n, m, seed, lo=0, hi=None, skew=False):
    rng = np.random.Generator(np.random.PCG64(seed))
    hi = n if hi is None else hi
    src = rng.integers(lo, hi, m)
    dst = rng.integers(lo, hi, m)
    if skew:
        src = lo + ((src - lo) * rng.random(m) ** 3).astype(np.int64)
        dst = lo + ((dst - lo) * rng.random(m) ** 4).astype(np.int64)
    return gg.Graph(n, src, dst, rng.integers(1, 1000, m), "rand")


def _one_source(n, m):
    rng = np.random.Generator(np.random.PCG64(3))
    g = _rand(n, m, 3)
    g.src[:] = n // 2
    g.w[:] = rng.integers(1, 50, m)
    return g


CASES = {
    "below": lambda: _rand(5000, M0 - 1, 1),
    "at the bound": lambda: _rand(5000, M0, 2),
    "one bucket": lambda: _rand(1024, M0 + 1, 4, skew=True),
    "bucket and one": lambda: _rand(1025, M0 + 8191, 5),
    "odd, skewed": lambda: _rand(262147, M0 + 5003, 6, skew=True),
    "one source": lambda: _one_source(3000, M0 + 77),
    "empty ends": lambda: _rand(3000001, M0 + 8192, 7, lo=1500000, hi=1600000, skew=True),
    "2^24 vertices": lambda: _rand(1 << 24, M0 + 3, 8, skew=True),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("kind,flags", [("coo", 0), ("coo", 1), ("coo", 2), ("coo", 4), ("csr", 0), ("csr", 2)])
def test_grouped_build(name, kind, flags):
    import paper_1903_01665_gb300 as fg
    g = CASES[name]()
    s = int(g.src[g.m // 2])
    d = oracle.sssp(g.n, g.src, g.dst, g.w, s)[1]
    lab = oracle.cc(g.n, g.src, g.dst)[1]
    outdeg = np.bincount(g.src, minlength=g.n)
    deg = outdeg + np.bincount(g.dst, minlength=g.n)
    with graph_handle(g, kind=kind, where="device", flags=flags) as h:
        for mode in (fg.FG_VERTEX_SYNC, fg.FG_EDGE_SYNC):
            got, _ = run(h, g.n, fg.FG_ALGO_SSSP, s, mode)
            np.testing.assert_array_equal(got, d)
            got, _ = run(h, g.n, fg.FG_ALGO_CC, 0, mode)
            np.testing.assert_array_equal(got, lab)
        _, p = fg.fg_select_plan(h, fg.FG_ALGO_SSSP)   # the default width shows the mean weight
        _, info = fg.fg_graph_info(h)
        assert info.n_zero_out == int((outdeg == 0).sum()) and info.n_isolated == int((deg == 0).sum())
        assert info.max_out_degree == int(outdeg.max())


@pytest.mark.parametrize("what", ["src", "dst", "weight", "both"])
def test_grouped_build_rejects(what):
    import paper_1903_01665_gb300 as fg
    g = _rand(4096, M0 + 9, 11)
    if what in ("src", "both"):
        g.src[-1] = 4096
    if what == "dst":
        g.dst[-1] = -1
    if what in ("weight", "both"):
        g.w[-1] = -3
    st, h = fg.fg_graph_create_coo(g.n, g.src, g.dst, g.w)
    assert h is None and st == (fg.FG_ERR_NEGATIVE_WEIGHT if what == "weight" else fg.FG_ERR_INVALID_ARG)
    st, h = fg.fg_graph_create_coo(g.n, np.abs(g.src) % 4096, np.abs(g.dst) % 4096, None)   # all ones
    fg.check(st)
    got, _ = run(h, g.n, fg.FG_ALGO_SSSP, 0, fg.FG_VERTEX_SYNC)
    np.testing.assert_array_equal(got, oracle.bfs(g.n, np.abs(g.src) % 4096, np.abs(g.dst) % 4096, 0)[1])
    fg.check(fg.fg_graph_destroy(h))
