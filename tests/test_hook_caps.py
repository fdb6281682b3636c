"""Components on renumbered graphs with a cap on rounds below the three that hooking and linking count as: the modes
propagate labels instead, as on graphs in their own order, and end where those do."""
import numpy as np
import pytest

import graphgen as gg
import paper_1903_01665_gb300 as fg
from tests.gpu_util import as_numpy, graph_handle, make_out

pytestmark = pytest.mark.gpu


def _edgeless(n):
    return gg.Graph(n, np.zeros(0, int), np.zeros(0, int), np.zeros(0, int), "edgeless")


def _pairs(n):
    """Edges from every odd vertex to the one before it: in-degrees of one and none, labels one hop away."""
    v = np.arange(1, n, 2)
    return gg.Graph(n, v, v - 1, np.ones(v.size, int), "pairs")


@pytest.mark.parametrize("mode", [fg.FG_VERTEX_ASYNC, fg.FG_BUCKET])
@pytest.mark.parametrize("make", [_edgeless, _pairs])
def test_caps(mode, make):
    n = 300
    g = make(n)
    want = np.arange(n) if g.src.size == 0 else np.arange(n) // 2 * 2
    rounds = {}
    for flags in (fg.FG_GRAPH_KEEP_IDS, fg.FG_GRAPH_RELABEL):
        with graph_handle(g, flags=flags) as h:
            for cap in (1, 2, 3, 0):
                out = make_out(n, "device", 99)
                st, stats = fg.fg_run(h, fg.FG_ALGO_CC, 0, out, mode, max_rounds=cap)
                assert st == fg.FG_OK if cap not in (1, 2) else st in (fg.FG_OK, fg.FG_ERR_TIMEOUT)
                rounds[flags, cap] = st
                np.testing.assert_array_equal(as_numpy(out), want if st == fg.FG_OK else np.full(n, 99))
                if st == fg.FG_OK:
                    assert stats.mode == mode
    # the smaller vertex of a pair is the one with an in-edge and renumbered first: both orders take as many rounds
    assert all(rounds[fg.FG_GRAPH_RELABEL, c] == rounds[fg.FG_GRAPH_KEEP_IDS, c] for c in (1, 2))
