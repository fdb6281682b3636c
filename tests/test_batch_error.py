"""A unit of a batch that ends with an error of its own (a worklist without room, made on the host) leaves the
units behind it in its team's queue alone."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1903_01665_gb300 as fg
from paper_1903_01665_gb300 import build as fgbuild
from tests.gpu_util import graph_handle

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
WORKLIST_BIT = 8


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    fg.load()
    so = str(tmp_path_factory.mktemp("batch_error") / "batch_error.so")
    where = os.path.dirname(fgbuild.LIB)
    subprocess.run([fgbuild._nvcc(), *fgbuild.ARCH, *fgbuild.NVCC_FLAGS, "-shared", "-cudart", "static",
                    os.path.join(HERE, "batch_error.cu"), "-o", so, fgbuild.LIB, "-Xlinker", "-rpath=" + where],
                   check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("team", [1, 2, 5, 64])
@pytest.mark.parametrize("flags", [fg.FG_GRAPH_KEEP_IDS, fg.FG_GRAPH_RELABEL])
def test_the_next_unit_runs(lib, team, flags):
    import torch
    g = gg.rmat(12, seed=3)
    s = int(gg.sources(g, 1, seed=4)[0])
    want = oracle.sssp(g.n, g.src, g.dst, g.w, s)[1]
    with graph_handle(g, flags=flags) as h:
        out = torch.full((g.n,), -7, dtype=torch.int32, device="cuda")
        status, done = (ctypes.c_int * 2)(), (ctypes.c_int * 2)()
        torch.cuda.synchronize()
        err = lib.run_two_units(ctypes.c_void_p(h), s, team,
                                ctypes.c_void_p(out.data_ptr()), status, done)
        assert err == 0
        assert status[0] == WORKLIST_BIT and not done[0]
        assert status[1] == 0 and done[1]
        np.testing.assert_array_equal(out.cpu().numpy(), want)
