"""FG_BUCKET's default width in the plan, which shows the sum of the weights (formed by the build's validation, its own
pass, or not at all without weights) and the bound between light and heavy edges: on graphs around the edge count from
which the build groups its edges, from edge lists and from rows."""
import numpy as np
import pytest

import graphgen as gg
import paper_1903_01665_gb300 as fg
from tests.gpu_util import graph_handle

pytestmark = pytest.mark.gpu
GROUPED = 1 << 20   # edges


def _shallow(m):
    """An R-MAT graph, renumbered: its rows are split where it has weights."""
    g = gg.rmat(17, edge_factor=9, seed=3)
    return gg.Graph(g.n, g.src[:m], g.dst[:m], g.w[:m], "rmat")


def _deep(m):
    """A grid of m edges or a few more among 2^21 vertices and more, most of them without edges if m is small."""
    side = 520
    while True:
        g = gg.grid(side, seed=5)
        if g.m >= m:
            break
        side += 8
    return gg.Graph(max(g.n, 1 << 21), g.src[:m], g.dst[:m], g.w[:m], "grid")


@pytest.mark.parametrize("kind", ["coo", "csr"])
@pytest.mark.parametrize("m", [GROUPED - 1, GROUPED, GROUPED + 777])
@pytest.mark.parametrize("make, weights", [(_shallow, True), (_deep, True), (_deep, False)])
def test_width(make, weights, m, kind):
    g = make(m)
    mean, deg = (int(g.w.astype(np.int64).sum()) / g.m if weights else 1.0), max(1.0, g.m / g.n)
    with graph_handle(g, kind=kind, weights=weights, where="device") as h:
        st, plan = fg.fg_select_plan(h, fg.FG_ALGO_SSSP)
        fg.check(st)
        assert plan.mode == fg.FG_BUCKET and plan.tuned == 0
        assert (plan.depth_est > 32) == (make is _deep)
        want = 2.0 * mean / deg if make is _shallow else 5.0 * mean * deg
        assert plan.delta == int(want + 0.5)
