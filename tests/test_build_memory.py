"""Graphs built where device memory suffices for the one-pass sort but not for the partition passes'
temporaries: the build does without them and gives the same graph.  The memory is bounded by a pool of limited
size, from which the library's allocations come while it is set."""
import contextlib
import ctypes

import pytest

import paper_1903_01665_gb300 as fg

pytestmark = pytest.mark.gpu
N, M = 1 << 18, 1 << 25
MARGIN = 96 << 20      # per-vertex arrays, queries, the pool's granularity; 6 bytes an edge are 192 MB


class _PoolProps(ctypes.Structure):
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int), ("location_type", ctypes.c_int),
                ("location_id", ctypes.c_int), ("security", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


@contextlib.contextmanager
def _memory_bound(limit):
    """The device's current memory pool: one of at most `limit` bytes."""
    cu = ctypes.CDLL("libcuda.so.1")
    pool, default = ctypes.c_void_p(), ctypes.c_void_p()
    props = _PoolProps(alloc_type=1, location_type=1, max_size=limit)   # pinned, device 0
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(default), 0) == 0
    assert cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) == 0
    assert cu.cuDeviceSetMemPool(0, pool) == 0
    try:
        yield
    finally:
        assert cu.cuDeviceSetMemPool(0, default) == 0
        assert cu.cuMemPoolDestroy(pool) == 0


@pytest.fixture(scope="module")
def edges():
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)

    def ids(power):
        return (torch.rand(M, generator=gen, device="cuda") ** power * N).int().clamp_(max=N - 1)
    return ids(2), ids(3), torch.randint(1, 1000, (M,), generator=gen, device="cuda", dtype=torch.int32)


def _results(edges, flags, calls):
    """Creates the graph and answers `calls`, in order."""
    import torch
    torch.cuda.synchronize()
    st, h = fg.fg_graph_create_coo(N, *edges, flags=flags)
    fg.check(st)
    outs = []
    try:
        for algo, mode in calls:
            out = torch.full((N,), -7, dtype=torch.int32, device="cuda")
            torch.cuda.synchronize()
            st, _ = fg.fg_run(h, algo, int(edges[0][0]), out, mode)
            fg.check(st)
            outs.append(out)
    finally:
        fg.check(fg.fg_graph_destroy(h))
    return outs


SSSP, CC = (fg.FG_ALGO_SSSP, fg.FG_VERTEX_SYNC), (fg.FG_ALGO_CC, fg.FG_VERTEX_SYNC)
BUCKET, PULL = (fg.FG_ALGO_SSSP, fg.FG_BUCKET), (fg.FG_ALGO_BFS, fg.FG_PULL)
CASES = {
    # flags, bytes an edge of the graph's arrays when the last call has run, calls
    "whole graph": (0, 28, [SSSP, BUCKET, CC]),
    "whole graph, own order": (fg.FG_GRAPH_KEEP_IDS, 28, [SSSP, CC]),
    "rows alone": (fg.FG_GRAPH_LAZY, 8, [SSSP, BUCKET]),
    "symmetrised view later": (fg.FG_GRAPH_LAZY, 28, [SSSP, CC]),
    "transposed view": (fg.FG_GRAPH_LAZY, 20, [PULL, SSSP]),
}


@pytest.mark.parametrize("name", list(CASES))
def test_build_in_little_memory(edges, name):
    import torch
    flags, per_edge, calls = CASES[name]
    want = _results(edges, flags, calls)
    with _memory_bound(per_edge * M + MARGIN):
        got = _results(edges, flags, calls)
    for g, w in zip(got, want):
        assert torch.equal(g, w)


def test_too_little_memory_is_reported(edges):
    import torch
    torch.cuda.synchronize()
    with _memory_bound(20 * M):
        st, h = fg.fg_graph_create_coo(N, *edges)
        assert st == fg.FG_ERR_OUT_OF_MEMORY and h is None
    _results(edges, 0, [SSSP])
