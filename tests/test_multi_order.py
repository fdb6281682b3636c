"""Which order a multi-source SSSP sweep takes on a renumbered graph: light edges first on large graphs whose edges are
mostly heavy, near-far on small ones and where half are light.  In a batch the near-far sweeps share a launch with the
BFS ones, the others have their own."""
import numpy as np
import pytest

import graphgen as gg
import paper_1903_01665_gb300 as fg
from tests.gpu_util import as_numpy, graph_handle, make_out, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale, weights, light", [(10, "uniform", False), (15, "uniform", False),
                                                   (16, "uniform", True), (16, "two values", False),
                                                   (20, "uniform", True), (20, "two values", False)])
def test_order(scale, weights, light):
    g = gg.rmat(scale, seed=3)
    if weights == "two values":
        rng = np.random.Generator(np.random.PCG64(1))
        g = gg.Graph(g.n, g.src, g.dst, np.where(rng.random(g.src.size) < 0.5, 1, 10000), "two")
    srcs = [int(s) for s in gg.sources(g, 2, seed=2)]
    with graph_handle(g, where="device") as h:
        qs = [(h, algo, s, make_out(g.n, "device"), fg.FG_VERTEX_SYNC)
              for algo in (fg.FG_ALGO_SSSP, fg.FG_ALGO_BFS) for s in srcs]
        st, _, _, bst = fg.fg_run_batch(qs, fuse_same_graph=True)
        fg.check(st)
        for _, algo, s, out, mode in qs:
            np.testing.assert_array_equal(as_numpy(out), run(h, g.n, algo, s, mode)[0])
        assert bst.launches == (2 if light else 1)
