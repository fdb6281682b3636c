"""FG_BUCKET SSSP on renumbered graphs with rows split by weight (light edges relaxed to a fixpoint below
the threshold, heavy ones once after it) against the oracle: widths far below and above the weights,
zero weights, rows of only light or only heavy edges, degrees around the classes' bounds, chains longer
than the threshold's doubling, sources without out-edges, batches, the overflow rule and the cap."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from tests.gpu_util import as_numpy, graph_handle, make_out, run

pytestmark = pytest.mark.gpu


def _chain(n, w_light, w_heavy):
    """A path whose weights alternate, beside a star that makes the in-degrees skewed."""
    p = np.arange(n - 1)
    w = np.where(p % 3 == 0, w_heavy, w_light)
    hub = np.arange(n, n + 3000)
    src = np.concatenate([p, hub, np.full(40, n - 1)])
    dst = np.concatenate([p + 1, np.full(3000, n), np.arange(n, n + 40)])
    w = np.concatenate([w, np.full(3000, 1), np.full(40, 999)])
    return gg.Graph(n + 3000, src, dst, w, "chain")


def _degrees():
    """Out-degrees 1, 31, 32, 1023, 1024, 2048, 2049 and 5000, weights 0..1000."""
    rng = np.random.Generator(np.random.PCG64(5))
    n, src = 6000, []
    for i, d in enumerate([1, 31, 32, 33, 1023, 1024, 1025, 2048, 2049, 5000]):
        src += [100 * i + k for k in range(3) for _ in range(d)]
    src = np.array(src + list(rng.integers(0, n, 20000)))
    return gg.Graph(n, src, rng.integers(0, n, src.size), rng.integers(0, 1001, src.size), "degrees")


CASES = {
    "rmat10": lambda: gg.rmat(10, seed=1),
    "rmat13": lambda: gg.rmat(13, seed=2),
    "rmat17": lambda: gg.rmat(17, seed=3),
    "zero weights": lambda: gg.rmat(11, seed=4, wlo=0, whi=300),
    "chain": lambda: _chain(400, 5, 700),
    "heavy chain": lambda: _chain(150, 900, 901),
    "degrees": _degrees,
    "hub": lambda: gg.hub(20000, 30000, 60000, seed=6),
}


@pytest.mark.parametrize("name", list(CASES))
def test_light_heavy(name):
    import paper_1903_01665_gb300 as fg
    g = CASES[name]()
    outdeg = np.bincount(g.src, minlength=g.n)
    srcs = [int(s) for s in gg.sources(g, 2, seed=3)] + [0, int(np.argmax(outdeg)), int(np.argmin(outdeg))]
    want = {s: oracle.sssp(g.n, g.src, g.dst, g.w, s)[1] for s in srcs}
    with graph_handle(g, flags=fg.FG_GRAPH_RELABEL) as h:
        for s in srcs:
            for delta in (0, 1, 7, 62, 500, 2**30, 2**31 - 1):
                got, st = run(h, g.n, fg.FG_ALGO_SSSP, s, fg.FG_BUCKET, delta=delta)
                np.testing.assert_array_equal(got, want[s], err_msg=f"{name} source {s} width {delta}")
                assert st.mode == fg.FG_BUCKET
            got, _ = run(h, g.n, fg.FG_ALGO_SSSP, s, fg.FG_BUCKET, blocks_per_sm=1, where="host")
            np.testing.assert_array_equal(got, want[s])
        outs = [make_out(g.n, "device") for _ in srcs]
        st, sts, stats, _ = fg.fg_run_batch([(h, fg.FG_ALGO_SSSP, s, o, fg.FG_BUCKET) for s, o in zip(srcs, outs)])
        fg.check(st)
        for s, o, x in zip(srcs, outs, stats):
            np.testing.assert_array_equal(as_numpy(o), want[s])
            assert x.mode == fg.FG_BUCKET


def test_light_heavy_limits():
    import paper_1903_01665_gb300 as fg
    g = _chain(60, 40, 800)
    g.w[10] = 2**31 - 300
    st_o, _ = oracle.sssp(g.n, g.src, g.dst, g.w, 0)
    with graph_handle(g, flags=fg.FG_GRAPH_RELABEL) as h:
        out = make_out(g.n, "device")
        st, _ = fg.fg_run(h, fg.FG_ALGO_SSSP, 0, out, fg.FG_BUCKET)
        assert st == fg.FG_ERR_OVERFLOW and (as_numpy(out) == -7).all()
        st, _ = fg.fg_run(h, fg.FG_ALGO_SSSP, 20, out, fg.FG_BUCKET, max_rounds=3)
        assert st == fg.FG_ERR_TIMEOUT and (as_numpy(out) == -7).all()
        st, _ = fg.fg_run(h, fg.FG_ALGO_SSSP, 0, out, fg.FG_BUCKET, inject_missing_arrival=1, wait_timeout_ms=50)
        assert st == fg.FG_ERR_TIMEOUT
        got, _ = run(h, g.n, fg.FG_ALGO_SSSP, 20, fg.FG_BUCKET)
        np.testing.assert_array_equal(got, oracle.sssp(g.n, g.src, g.dst, g.w, 20)[1])
