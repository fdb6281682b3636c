"""Pull rounds of the multi-source BFS (renumbered graphs with their symmetrised view) against the oracle:
in-degrees around the lane's own tries, the warp's batches and the chunk size, hubs that some sources
never reach, sources in components of their own, a lazy graph (which only pushes), fused batches."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from tests.gpu_util import as_numpy, graph_handle, make_out
from tests.test_pull_early import _in_degrees

pytestmark = pytest.mark.gpu


def _island(g, seed):
    """g beside a path that one source starts on."""
    n, p = g.n, 300
    src = np.concatenate([g.src, np.arange(n, n + p - 1)])
    dst = np.concatenate([g.dst, np.arange(n + 1, n + p)])
    return gg.Graph(n + p, src, dst, np.ones(src.size, np.int32), g.name + "+path")


@pytest.mark.parametrize("case", ["in-degrees 1", "in-degrees 40", "rmat 14", "rmat 16"])
@pytest.mark.parametrize("lazy", [False, True])
def test_multi_pull(case, lazy):
    import paper_1903_01665_gb300 as fg
    g = {"in-degrees 1": lambda: _in_degrees(3, 1), "in-degrees 40": lambda: _in_degrees(4, 40),
         "rmat 14": lambda: gg.rmat(14, seed=6), "rmat 16": lambda: gg.rmat(16, seed=7)}[case]()
    g = _island(g, 1)
    srcs = [0] + [int(s) for s in gg.sources(g, 5, seed=8)] + [g.n - 300, g.n - 1]
    want = [oracle.bfs(g.n, g.src, g.dst, s)[1] for s in srcs]
    flags = fg.FG_GRAPH_RELABEL | (fg.FG_GRAPH_LAZY if lazy else 0)
    with graph_handle(g, flags=flags) as h:
        for k in (8, 3, 1):
            for kw in ({}, {"blocks_per_sm": 1}):
                outs = [make_out(g.n, "device" if j != 1 else "host") for j in range(k)]
                st, sts, _ = fg.fg_run_multi(h, fg.FG_ALGO_BFS, srcs[:k], outs, **kw)
                fg.check(st)
                for o, w, s in zip(outs, want, srcs):
                    np.testing.assert_array_equal(as_numpy(o), w, err_msg=f"{case} source {s} k {k}")
        outs = [make_out(g.n, "device") for _ in srcs]
        st, _, _, _ = fg.fg_run_batch([(h, fg.FG_ALGO_BFS, s, o, fg.FG_AUTO) for s, o in zip(srcs, outs)],
                                      fuse_same_graph=True)
        fg.check(st)
        for o, w in zip(outs, want):
            np.testing.assert_array_equal(as_numpy(o), w)
