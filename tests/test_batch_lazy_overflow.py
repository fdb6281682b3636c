"""The overflow check of a batch's single-source query reads the edge sources: on a graph that was created without them
they are built first."""
import numpy as np
import pytest

import graphgen as gg
import paper_1903_01665_gb300 as fg
from tests.gpu_util import as_numpy, graph_handle, make_out

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [fg.FG_VERTEX_SYNC, fg.FG_VERTEX_ASYNC, fg.FG_BUCKET])
@pytest.mark.parametrize("flags", [0, fg.FG_GRAPH_RELABEL])
def test_overflow_on_a_lazy_graph(mode, flags):
    g = gg.path(3, weights=[2**30, 2**30])
    with graph_handle(g, flags=fg.FG_GRAPH_LAZY | flags) as h:
        outs = [make_out(g.n, "device"), make_out(g.n, "host")]
        st, sts, _, _ = fg.fg_run_batch([(h, fg.FG_ALGO_SSSP, s, o, mode) for s, o in enumerate(outs)])
        assert st == fg.FG_ERR_OVERFLOW and sts == [fg.FG_ERR_OVERFLOW, fg.FG_OK]
        np.testing.assert_array_equal(as_numpy(outs[1]), [fg.FG_INF, 0, 2**30])
