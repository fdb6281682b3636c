"""Pull rounds of the multi-source BFS on graphs whose hubs lie among other vertices in the renumbered order
(many out-edges, few in-edges): in one round a hub's chunk and its neighbours in the same four-byte word of
the reached-by masks are claimed at the same time."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from tests.gpu_util import as_numpy, graph_handle, make_out

pytestmark = pytest.mark.gpu


def _hubs_among_others(seed, n=24000, k=8, first=2500, hub_every=97):
    """Sources 0..k-1 reach `first` vertices each in one step, and from there every later vertex over its
    four to seven in-edges in the next; every hub_every-th of those has 1,500 out-edges (into the first)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    nf = 2 * first
    a_src, a_dst = [], []
    for s in range(k):
        to = k + rng.choice(nf, first, replace=False)
        a_src.append(np.full(first, s))
        a_dst.append(to)
    later = np.arange(k + nf, n)
    cnt = rng.integers(4, 8, later.size)
    a_dst.append(np.repeat(later, cnt))
    a_src.append(k + rng.integers(0, nf, cnt.sum()))
    hubs = later[::hub_every]
    a_src.append(np.repeat(hubs, 1500))
    a_dst.append(k + rng.integers(0, nf, hubs.size * 1500))
    src, dst = np.concatenate(a_src), np.concatenate(a_dst)
    return gg.Graph(n, src, dst, np.ones(src.size, np.int32), "hubs among others")


@pytest.mark.parametrize("hub_every", [3, 97])
def test_hubs_beside_others_in_a_word(hub_every):
    import paper_1903_01665_gb300 as fg
    g = _hubs_among_others(5, hub_every=hub_every)
    srcs = list(range(8))
    want = [oracle.bfs(g.n, g.src, g.dst, s)[1] for s in srcs]
    with graph_handle(g, flags=fg.FG_GRAPH_RELABEL) as h:
        for k in (8, 5):
            for kw in ({}, {"blocks_per_sm": 1}):
                for _ in range(5):
                    outs = [make_out(g.n, "device") for _ in range(k)]
                    st, _, _ = fg.fg_run_multi(h, fg.FG_ALGO_BFS, srcs[:k], outs, **kw)
                    fg.check(st)
                    for o, w, s in zip(outs, want, srcs):
                        np.testing.assert_array_equal(as_numpy(o), w, err_msg=f"source {s} of {k}")
        outs = [make_out(g.n, "device") for _ in srcs]
        st, _, stats, _ = fg.fg_run_batch([(h, fg.FG_ALGO_BFS, s, o, fg.FG_VERTEX_SYNC) for s, o in zip(srcs, outs)],
                                          fuse_same_graph=True)
        fg.check(st)
        assert stats[0].pull_rounds > 0   # the sweep does pull on this graph
        for o, w in zip(outs, want):
            np.testing.assert_array_equal(as_numpy(o), w)
