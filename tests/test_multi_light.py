"""Multi-source SSSP in the light-heavy order (renumbered graphs with split rows) against the oracle:
sources that enter the hubs at different distances, widths far below and above the weights, repeats, a
source without out-edges, one slot overflowing, few CTAs, fused batches."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from tests.gpu_util import as_numpy, graph_handle, make_out
from tests.test_light_heavy import CASES, _chain

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", list(CASES))
def test_multi_light(name):
    import paper_1903_01665_gb300 as fg
    g = CASES[name]()
    outdeg = np.bincount(g.src, minlength=g.n)
    srcs = [int(s) for s in gg.sources(g, 5, seed=4)] + [int(np.argmax(outdeg)), int(np.argmin(outdeg))]
    srcs = (srcs + [srcs[0]])[:8]
    want = [oracle.sssp(g.n, g.src, g.dst, g.w, s)[1] for s in srcs]
    with graph_handle(g, flags=fg.FG_GRAPH_RELABEL) as h:
        for k, kw in ((8, {}), (8, {"delta": 1}), (3, {"delta": 500}), (2, {"delta": 2**31 - 1}), (8, {"blocks_per_sm": 1}),
                      (1, {"delta": 2**30})):
            k = min(k, len(srcs))
            outs = [make_out(g.n, "device" if j % 3 else "host") for j in range(k)]
            st, sts, _ = fg.fg_run_multi(h, fg.FG_ALGO_SSSP, srcs[:k], outs, **kw)
            fg.check(st)
            for o, w, s in zip(outs, want, srcs):
                np.testing.assert_array_equal(as_numpy(o), w, err_msg=f"{name} source {s} k {k} {kw}")
        outs = [make_out(g.n, "device") for _ in srcs]
        st, _, _, _ = fg.fg_run_batch([(h, fg.FG_ALGO_SSSP, s, o, fg.FG_AUTO) for s, o in zip(srcs, outs)],
                                      fuse_same_graph=True)
        fg.check(st)
        for o, w in zip(outs, want):
            np.testing.assert_array_equal(as_numpy(o), w)


def test_multi_light_overflow_and_cap():
    import paper_1903_01665_gb300 as fg
    g = _chain(60, 40, 800)
    g.w[10] = 2**31 - 300
    with graph_handle(g, flags=fg.FG_GRAPH_RELABEL) as h:
        srcs = [0, 20, 40]
        outs = [make_out(g.n, "device") for _ in srcs]
        st, sts, _ = fg.fg_run_multi(h, fg.FG_ALGO_SSSP, srcs, outs)
        assert st == fg.FG_ERR_OVERFLOW and sts == [fg.FG_ERR_OVERFLOW, fg.FG_OK, fg.FG_OK]
        assert (as_numpy(outs[0]) == -7).all()
        for s, o in list(zip(srcs, outs))[1:]:
            np.testing.assert_array_equal(as_numpy(o), oracle.sssp(g.n, g.src, g.dst, g.w, s)[1])
        st, sts, _ = fg.fg_run_multi(h, fg.FG_ALGO_SSSP, [20, 40], outs[1:], max_rounds=2)
        assert st == fg.FG_ERR_TIMEOUT
