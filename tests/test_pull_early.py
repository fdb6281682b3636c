"""BFS pull rounds with early exit against the oracle: in-degrees around the lanes' own tries (1-5), the
class bounds (31-33, 1023-1025) and the chunk size (2048, 2049, 4097), parents only at the end of a list,
unreachable hubs, graphs renumbered or not."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from tests.gpu_util import graph_handle, run

pytestmark = pytest.mark.gpu
DEGREES = [1, 2, 3, 4, 5, 6, 31, 32, 33, 36, 37, 1023, 1024, 1025, 2047, 2048, 2049, 4097]


def _in_degrees(seed, frontier):
    """Targets of each in-degree; `frontier` of each list's sources are reachable from vertex 0 in one
    step, at random places, the others are not reachable at all."""
    rng = np.random.Generator(np.random.PCG64(seed))
    n, reach, dead = 20000, np.arange(1, 6001), np.arange(6001, 12001)
    src, dst = [np.zeros(reach.size, np.int64)], [reach]
    v = 12001
    for d in DEGREES:
        for k in range(4):
            u = rng.choice(dead, d)
            f = min(d, frontier if k % 2 else 0)
            u[rng.choice(d, f, replace=False)] = rng.choice(reach, f)
            src.append(u)
            dst.append(np.full(d, v))
            v += 1
    src.append(rng.integers(12001, v, 3000))
    dst.append(rng.integers(v, n, 3000))
    return gg.Graph(n, np.concatenate(src), np.concatenate(dst), np.ones(sum(map(len, src)), np.int32),
                    "in-degrees")


@pytest.mark.parametrize("frontier", [1, 2, 40])
@pytest.mark.parametrize("flags", ["relabel", "keep"])
def test_pull_early_exit(frontier, flags):
    import paper_1903_01665_gb300 as fg
    fl = fg.FG_GRAPH_RELABEL if flags == "relabel" else fg.FG_GRAPH_KEEP_IDS
    for g in (_in_degrees(7 + frontier, frontier), gg.rmat(14, seed=frontier), gg.er(9000, 90000, seed=frontier)):
        s = 0 if g.name == "in-degrees" else int(gg.sources(g, 1, seed=2)[0])
        want = oracle.bfs(g.n, g.src, g.dst, s)[1]
        with graph_handle(g, flags=fl) as h:
            got, st = run(h, g.n, fg.FG_ALGO_BFS, s, fg.FG_PULL)
            np.testing.assert_array_equal(got, want)
            assert st.pull_rounds > 0
            got, _ = run(h, g.n, fg.FG_ALGO_BFS, s, fg.FG_PULL, blocks_per_sm=1)
            np.testing.assert_array_equal(got, want)
