"""A cap on rounds that is enough for a mode's own rounds is enough for the call, whatever order the graph would
otherwise be taken in (light and heavy edges, hooking and linking), and the automatic choice keeps to it."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1903_01665_gb300 as fg
from tests.gpu_util import as_numpy, graph_handle, make_out, run

pytestmark = pytest.mark.gpu


def _path(n, seed):
    """A path with a few heavy shortcuts, so that its rows are split by weight."""
    rng = np.random.Generator(np.random.PCG64(seed))
    src = np.concatenate([np.arange(n - 1), rng.integers(0, n, 40)])
    dst = np.concatenate([np.arange(1, n), rng.integers(0, n, 40)])
    w = np.concatenate([rng.integers(1, 200, n - 1), rng.integers(150000, 300000, 40)])
    return gg.Graph(n, src, dst, w, "path")


def _star(leaves, kind):
    """Edges into the hub (0), out of it, or out of it with two loops at it."""
    hub, leaf = np.zeros(leaves, int), np.arange(1, leaves + 1)
    src, dst = (leaf, hub) if kind == "in" else (hub, leaf)
    if kind == "out, loops":
        src, dst = np.concatenate([src, [0, 0]]), np.concatenate([dst, [0, 0]])
    return gg.Graph(leaves + 1, src, dst, np.ones(src.size, int), "star")


@pytest.mark.parametrize("n", [150, 900])
def test_bucket_with_a_cap_of_n_plus_2(n):
    g = _path(n, n)
    want = oracle.sssp(g.n, g.src, g.dst, g.w, 0)[1]
    with graph_handle(g, flags=fg.FG_GRAPH_RELABEL) as h:
        for cap in (0, n + 2, 8 * n + 63, 8 * n + 64):
            got, _ = run(h, g.n, fg.FG_ALGO_SSSP, 0, fg.FG_BUCKET, max_rounds=cap)
            np.testing.assert_array_equal(got, want, err_msg=f"cap {cap}")
        out = make_out(g.n, "device", 99)
        assert fg.fg_run(h, fg.FG_ALGO_SSSP, 0, out, fg.FG_BUCKET, max_rounds=2)[0] == fg.FG_ERR_TIMEOUT
        assert (as_numpy(out) == 99).all()


def test_multi_with_the_cap_of_other_graphs():
    g = _path(400, 7)
    srcs = [0, 3, 399]
    with graph_handle(g, flags=fg.FG_GRAPH_RELABEL) as h:
        for cap in (0, 2 * 3 * 400 + 2, 8 * 3 * 400 + 63, 8 * 3 * 400 + 64):
            outs = [make_out(g.n, "device") for _ in srcs]
            st, _, _ = fg.fg_run_multi(h, fg.FG_ALGO_SSSP, srcs, outs, max_rounds=cap)
            fg.check(st)
            for o, s in zip(outs, srcs):
                np.testing.assert_array_equal(as_numpy(o), oracle.sssp(g.n, g.src, g.dst, g.w, s)[1])
        outs = [make_out(g.n, "device") for _ in srcs]
        assert fg.fg_run_multi(h, fg.FG_ALGO_SSSP, srcs, outs, max_rounds=2)[0] == fg.FG_ERR_TIMEOUT


@pytest.mark.parametrize("mode", [fg.FG_EDGE_SYNC, fg.FG_AUTO])
def test_components_with_a_small_cap(mode):
    # the hub is renumbered first by its in-edges, and last without any: then its label takes a generation
    # to reach it and another to come back
    for kind, enough in (("in", 2), ("out", 3), ("out, loops", 2)):
        g = _star(700, kind)
        with graph_handle(g, flags=fg.FG_GRAPH_RELABEL) as h:
            for cap in (1, 2, 3, 0):
                out = make_out(g.n, "device", 99)
                st, stats = fg.fg_run(h, fg.FG_ALGO_CC, 0, out, mode, max_rounds=cap)
                if cap and cap < enough:
                    assert st == fg.FG_ERR_TIMEOUT and (as_numpy(out) == 99).all()
                else:
                    fg.check(st)
                    assert (as_numpy(out) == 0).all() and (not cap or stats.rounds <= cap)


def test_auto_with_the_rounds_of_the_edge_form():
    g = gg.rmat(17, seed=9)
    s = int(gg.sources(g, 1, seed=2)[0])
    want = oracle.sssp(g.n, g.src, g.dst, g.w, s)[1]
    with graph_handle(g) as h:
        got, free = run(h, g.n, fg.FG_ALGO_SSSP, s, fg.FG_AUTO)
        np.testing.assert_array_equal(got, want)
        _, edge = run(h, g.n, fg.FG_ALGO_SSSP, s, fg.FG_EDGE_ASYNC)
        cap = edge.rounds + 3   # the generations vary a little from run to run
        assert free.mode == fg.FG_BUCKET and free.rounds > cap
        got, stats = run(h, g.n, fg.FG_ALGO_SSSP, s, fg.FG_AUTO, max_rounds=cap)
        np.testing.assert_array_equal(got, want)
        assert stats.mode == fg.FG_EDGE_ASYNC
