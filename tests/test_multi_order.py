"""Which order a multi-source SSSP sweep takes on a renumbered graph: light edges first on large graphs whose edges are
mostly heavy, near-far (what a cap below the other order's rounds selects) on small ones and where half are light."""
import numpy as np
import pytest

import graphgen as gg
import paper_1903_01665_gb300 as fg
from tests.gpu_util import as_numpy, graph_handle, make_out, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale, weights, light", [(10, "uniform", False), (14, "uniform", False),
                                                   (20, "uniform", True), (20, "two values", False)])
def test_order(scale, weights, light):
    g = gg.rmat(scale, seed=3)
    if weights == "two values":
        rng = np.random.Generator(np.random.PCG64(1))
        g = gg.Graph(g.n, g.src, g.dst, np.where(rng.random(g.src.size) < 0.5, 1, 10000), "two")
    srcs = [int(s) for s in gg.sources(g, 4, seed=2)]
    with graph_handle(g, where="device") as h:
        def sweep(**kw):
            outs = [make_out(g.n, "device") for _ in srcs]
            st, _, stats = fg.fg_run_multi(h, fg.FG_ALGO_SSSP, srcs, outs, **kw)
            fg.check(st)
            for o, s in zip(outs, srcs):
                np.testing.assert_array_equal(as_numpy(o), run(h, g.n, fg.FG_ALGO_SSSP, s, fg.FG_VERTEX_SYNC)[0])
            return stats.rounds
        own, near_far = sweep(), sweep(max_rounds=8 * 4 * g.n + 63)
        assert (own > 1.5 * near_far) == light
