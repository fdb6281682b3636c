"""Two host threads that create graphs of different shapes at the same time, and build their transposed
views: a build of one shape must not disturb a launch of the other's (the shared memory that the grouping
kernels may use is a property of the kernel, not of the caller)."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROUNDS = 120


def _edges(n, seed):
    import torch
    rng = np.random.Generator(np.random.PCG64(seed))
    m = (1 << 20) + 37
    src = (n * rng.random(m) ** 2).astype(np.int32)
    dst = (n * rng.random(m) ** 3).astype(np.int32)
    w = rng.integers(1, 1000, m).astype(np.int32)
    return [torch.from_numpy(x).cuda() for x in (src, dst, w)]


def _bfs_of_new_graph(n, edges, out):
    import paper_1903_01665_gb300 as fg
    st, h = fg.fg_graph_create_coo(n, *edges)
    fg.check(st)
    try:
        fg.check(fg.fg_bfs(h, int(edges[0][0]), out, fg.FG_PULL))   # builds the transposed view
    finally:
        fg.check(fg.fg_graph_destroy(h))


def test_builds_of_two_shapes_from_two_threads():
    import torch
    shapes = [[1 << 22], [1 << 20, 1024, 1 << 14]]
    edges = {n: _edges(n, n) for s in shapes for n in s}
    want = {}
    for n, e in edges.items():
        want[n] = torch.empty(n, dtype=torch.int32, device="cuda")
        _bfs_of_new_graph(n, e, want[n])
    errors = []

    def work(sizes):
        try:
            torch.cuda.set_device(0)
            for k in range(ROUNDS):
                n = sizes[k % len(sizes)]
                out = torch.full((n,), -7, dtype=torch.int32, device="cuda")
                torch.cuda.synchronize()
                _bfs_of_new_graph(n, edges[n], out)
                if not torch.equal(out, want[n]):
                    errors.append(f"n = {n}: another result")
        except Exception as e:   # noqa: BLE001 - reported by the main thread
            errors.append(str(e))

    threads = [threading.Thread(target=work, args=(s,)) for s in shapes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
