"""The dense scans and short worklists take 8, 16, 32 or 128 vertices a warp step by the number of
vertices and warps: every mode and the multi-source sweeps against the oracle just below, at and
above each of those sizes (one CTA per SM: sms * 8 warps)."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from tests.gpu_util import MODES, make_out, as_numpy, graph_handle, run


@pytest.mark.gpu
@pytest.mark.parametrize("per_warp,off", [(8, -1), (8, 1), (16, 0), (16, 1), (128, -1), (128, 0), (128, 3)])
def test_scan_step_edges(per_warp, off):
    import torch

    import paper_1903_01665_gb300 as fg
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = sms * 8 * per_warp + off
    g = gg.er(n, 6 * n + 5, seed=per_warp * 10 + off + 1)
    srcs = [int(s) for s in gg.sources(g, 3, seed=5)]
    dist = [oracle.sssp(g.n, g.src, g.dst, g.w, s)[1] for s in srcs]
    lev = [oracle.bfs(g.n, g.src, g.dst, s)[1] for s in srcs]
    with graph_handle(g, where="device") as h:
        for mode in MODES:
            for algo, want in ((fg.FG_ALGO_SSSP, dist[0]), (fg.FG_ALGO_BFS, lev[0])):
                got, _ = run(h, g.n, algo, srcs[0], mode, blocks_per_sm=1)
                np.testing.assert_array_equal(got, want, err_msg=f"n={n} algo {algo} mode {mode}")
        for algo, want in ((fg.FG_ALGO_SSSP, dist), (fg.FG_ALGO_BFS, lev)):
            outs = [make_out(g.n, "device") for _ in srcs]
            st, sts, _ = fg.fg_run_multi(h, algo, srcs, outs, blocks_per_sm=1)
            fg.check(st)
            for o, w in zip(outs, want):
                np.testing.assert_array_equal(as_numpy(o), w)
