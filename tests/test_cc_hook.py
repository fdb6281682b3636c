"""Components by hooking and linking (the worklist modes on renumbered graphs) against the oracle, on
the shapes that it treats differently: several large trees, hubs outside the largest component, long
chains in id order and in a random order, rows just around the sampled neighbours, isolated vertices."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from tests.gpu_util import graph_handle, run

pytestmark = pytest.mark.gpu


def _join(*parts, seed=None):
    """Disjoint union of graphs, ids shuffled if a seed is given."""
    n = sum(p.n for p in parts)
    src, dst, base = [], [], 0
    for p in parts:
        src.append(p.src.astype(np.int64) + base)
        dst.append(p.dst.astype(np.int64) + base)
        base += p.n
    src, dst = np.concatenate(src), np.concatenate(dst)
    if seed is not None:
        perm = np.random.Generator(np.random.PCG64(seed)).permutation(n)
        src, dst = perm[src], perm[dst]
    return gg.Graph(n, src, dst, np.ones(src.size, np.int32), "join")


def _cases():
    yield "one", gg.Graph(1, [], [], [], "one")
    yield "isolated", gg.Graph(777, [], [], [], "isolated")
    yield "long path in order, star", _join(gg.path(200000), gg.star(5000))
    yield "long path shuffled, star", _join(gg.path(60000), gg.star(3000), seed=3)
    yield "two equal rmat", _join(gg.rmat(12, seed=1), gg.rmat(12, seed=2))
    yield "two equal rmat shuffled", _join(gg.rmat(12, seed=1), gg.rmat(12, seed=2), gg.path(500), seed=4)
    yield "hub beside a larger grid", _join(gg.star(2500), gg.full_grid(150, 150))
    yield "small cliques around the samples", gg.disjoint_cliques([1, 2, 3, 4, 5, 6, 31, 32, 33, 34, 63, 64, 65, 66,
                                                                   255, 256, 257, 258, 1025, 1])
    yield "rmat 14", gg.rmat(14, seed=9)


@pytest.mark.parametrize("name,g", list(_cases()), ids=[c[0] for c in _cases()])
def test_cc_hook_link(name, g):
    import torch

    import paper_1903_01665_gb300 as fg
    want = oracle.cc(g.n, g.src, g.dst)[1]
    with graph_handle(g, flags=fg.FG_GRAPH_RELABEL) as h:
        for mode in (fg.FG_VERTEX_ASYNC, fg.FG_BUCKET):
            got, st = run(h, g.n, fg.FG_ALGO_CC, 0, mode)
            np.testing.assert_array_equal(got, want)
            assert st.rounds == 3
            s, _ = fg.fg_run(h, fg.FG_ALGO_CC, 0, torch.empty(g.n, dtype=torch.int32, device="cuda"), mode,
                             max_rounds=2)
            assert s == fg.FG_ERR_TIMEOUT
        out = torch.empty(g.n, dtype=torch.int32, device="cuda")
        s, sts, _, _ = fg.fg_run_batch([(h, fg.FG_ALGO_CC, 0, out, fg.FG_VERTEX_ASYNC)])
        fg.check(s)
        np.testing.assert_array_equal(out.cpu().numpy(), want)
