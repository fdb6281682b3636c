"""SSSP on renumbered graphs that are deep all the same (an R-MAT graph joined to a grid): the light-heavy order, which
would need hundreds of generations there, ends at its limit and the near-far order of other graphs runs, at once from
then on or once the depth estimate is known; results are the oracle's throughout."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1903_01665_gb300 as fg
from tests.gpu_util import as_numpy, graph_handle, make_out, run
from tests.test_build_memory import _memory_bound

pytestmark = pytest.mark.gpu
LIMIT = 128   # generations of the light-heavy order


def _deep(scale=12, side=110):
    a, b = gg.rmat(scale, seed=1), gg.grid(side, seed=2)
    at = np.array([0, a.n])
    src = np.concatenate([a.src, b.src + a.n, at])
    dst = np.concatenate([a.dst, b.dst + a.n, at[::-1]])
    return gg.Graph(a.n + b.n, src, dst, np.concatenate([a.w, b.w, [1, 1]]), "deep")


@pytest.fixture(scope="module")
def deep():
    g = _deep()
    srcs = [int(s) for s in gg.sources(g, 3, seed=5)] + [0, g.n - 1]
    return g, srcs, [oracle.sssp(g.n, g.src, g.dst, g.w, s)[1] for s in srcs]


def _near_far_rounds(h, g, s):
    return run(h, g.n, fg.FG_ALGO_SSSP, s, fg.FG_BUCKET, max_rounds=8 * g.n + 63)[1].rounds


@pytest.mark.parametrize("where", ["device", "host"])
def test_bucket(deep, where):
    g, srcs, want = deep
    with graph_handle(g, flags=fg.FG_GRAPH_RELABEL) as h:
        plain = _near_far_rounds(h, g, srcs[0])
        for _ in range(2):
            for s, w in zip(srcs, want):
                got, stats = run(h, g.n, fg.FG_ALGO_SSSP, s, fg.FG_BUCKET, where=where)
                np.testing.assert_array_equal(got, w)
                assert stats.mode == fg.FG_BUCKET
        assert run(h, g.n, fg.FG_ALGO_SSSP, srcs[0], fg.FG_BUCKET)[1].rounds <= 1.5 * plain


def test_known_depth(deep):
    g, srcs, want = deep
    with graph_handle(g, flags=fg.FG_GRAPH_RELABEL) as h:
        st, plan = fg.fg_select_plan(h, fg.FG_ALGO_SSSP)
        fg.check(st)
        assert plan.depth_est > 32
        plain = _near_far_rounds(h, g, srcs[0])
        before = fg.fg_kernel_launches()
        got, stats = run(h, g.n, fg.FG_ALGO_SSSP, srcs[0], fg.FG_BUCKET)
        np.testing.assert_array_equal(got, want[0])
        assert stats.rounds <= 1.5 * plain
        assert fg.fg_kernel_launches() - before == 2   # one fixpoint, and the output to original order


@pytest.mark.parametrize("k", [2, 5])
def test_multi(deep, k):
    g, srcs, want = deep
    with graph_handle(g, flags=fg.FG_GRAPH_RELABEL) as h:
        for delta in (0, 40, 0):   # with a width of the caller's the light-heavy order also on a small graph
            outs = [make_out(g.n, "host" if j == 1 else "device") for j in range(k)]
            st, sts, stats = fg.fg_run_multi(h, fg.FG_ALGO_SSSP, srcs[:k], outs, delta=delta)
            fg.check(st)
            assert sts == [fg.FG_OK] * k
            for o, w in zip(outs, want):
                np.testing.assert_array_equal(as_numpy(o), w)


def test_sweeps_of_a_large_graph():
    g = _deep(20, 250)
    srcs = [int(s) for s in gg.sources(g, 4, seed=5)]
    with graph_handle(g, where="device") as h:
        want = [run(h, g.n, fg.FG_ALGO_SSSP, s, fg.FG_VERTEX_SYNC)[0] for s in srcs]
        rounds = []
        for _ in range(2):
            outs = [make_out(g.n, "host" if j == 1 else "device") for j in range(4)]
            st, _, stats = fg.fg_run_multi(h, fg.FG_ALGO_SSSP, srcs, outs)
            fg.check(st)
            rounds.append(stats.rounds)
            for o, w in zip(outs, want):
                np.testing.assert_array_equal(as_numpy(o), w)
        near_far = fg.fg_run_multi(h, fg.FG_ALGO_SSSP, srcs, outs, max_rounds=8 * 4 * g.n + 63)[2].rounds
        assert max(rounds) <= 1.5 * near_far
    with graph_handle(g, where="device") as h:   # not known yet: the batch meets the limit itself
        outs = [make_out(g.n, ("host", "device", "pinned")[j % 3]) for j in range(4)]
        st, sts, stats, _ = fg.fg_run_batch([(h, fg.FG_ALGO_SSSP, s, o, fg.FG_VERTEX_SYNC) for s, o in zip(srcs, outs)],
                                            fuse_same_graph=True)
        fg.check(st)
        for o, w in zip(outs, want):
            np.testing.assert_array_equal(as_numpy(o), w)
        assert all(s.mode == -1 and s.rounds <= 1.5 * near_far for s in stats)


def test_a_far_source_alone_does_not_make_a_graph_deep():
    """A long path into an R-MAT graph: its end takes many generations, the others few."""
    a, n = gg.rmat(12, seed=1), 600
    p = a.n + np.arange(n - 1)
    g = gg.Graph(a.n + n, np.concatenate([a.src, p, [a.n + n - 1]]), np.concatenate([a.dst, p + 1, [0]]),
                 np.concatenate([a.w, np.full(n, 3)]), "tail")
    near, far = int(gg.sources(a, 1, seed=4)[0]), a.n
    with graph_handle(g, flags=fg.FG_GRAPH_RELABEL) as h:
        rounds = []
        for s in (near, far, near, near):
            got, stats = run(h, g.n, fg.FG_ALGO_SSSP, s, fg.FG_BUCKET)
            np.testing.assert_array_equal(got, oracle.sssp(g.n, g.src, g.dst, g.w, s)[1])
            rounds.append(stats.rounds)
        # the near-far order in the third, the light-heavy one, which takes more generations, in the others
        assert rounds[1] > 32 and rounds[2] < rounds[0] and rounds[3] > rounds[2]
        run(h, g.n, fg.FG_ALGO_SSSP, far, fg.FG_BUCKET)
        assert run(h, g.n, fg.FG_ALGO_SSSP, near, fg.FG_EDGE_ASYNC)[1].rounds <= 32   # any other mode tells, too
        assert run(h, g.n, fg.FG_ALGO_SSSP, near, fg.FG_BUCKET)[1].rounds > rounds[2]


@pytest.mark.parametrize("graph", [False, True])
def test_batch(deep, graph):
    g, srcs, want = deep
    other = gg.rmat(10, seed=9)
    exp = oracle.sssp(other.n, other.src, other.dst, other.w, 1)[1]
    with graph_handle(g, flags=fg.FG_GRAPH_RELABEL) as h, graph_handle(other, flags=fg.FG_GRAPH_RELABEL) as ho:
        for _ in range(2):
            outs = [make_out(g.n, ("device", "host", "pinned")[j % 3]) for j in range(len(srcs))]
            last = make_out(other.n, "host")
            qs = [(h, fg.FG_ALGO_SSSP, s, o, fg.FG_BUCKET) for s, o in zip(srcs, outs)]
            qs.append((ho, fg.FG_ALGO_SSSP, 1, last, fg.FG_BUCKET))
            st, sts, stats, _ = fg.fg_run_batch(qs, use_cuda_graph=graph)
            fg.check(st)
            for o, w in zip(outs, want):
                np.testing.assert_array_equal(as_numpy(o), w)
            np.testing.assert_array_equal(last, exp)
            assert all(s.mode == fg.FG_BUCKET for s in stats) and stats[-1].rounds <= LIMIT


def test_near_far_without_the_memory_for_it(deep):
    """The near-far order takes 28 bytes a vertex, the other 9: where only that is there, it runs after all."""
    import torch
    g, srcs, _ = deep
    g = gg.Graph(6 << 20, g.src, g.dst, g.w, "deep, isolated vertices")
    want = oracle.sssp(g.n, g.src, g.dst, g.w, srcs[0])[1]
    with graph_handle(g, flags=fg.FG_GRAPH_RELABEL, where="device") as h:
        st, plan = fg.fg_select_plan(h, fg.FG_ALGO_SSSP)
        fg.check(st)
        assert plan.depth_est > 32
        out = make_out(g.n, "device")
        torch.cuda.synchronize()
        rounds = []
        for limit in (96 << 20, 512 << 20):
            with _memory_bound(limit):
                st, stats = fg.fg_run(h, fg.FG_ALGO_SSSP, srcs[0], out, fg.FG_BUCKET)
                fg.check(st)
            rounds.append(stats.rounds)
            np.testing.assert_array_equal(as_numpy(out), want)
        assert rounds[0] > LIMIT > 0 and rounds[0] > rounds[1]
