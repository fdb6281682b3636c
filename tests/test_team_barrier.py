"""The team barrier when a wait runs out: the CTA that arrives last, after another one gave up, learns of it
from the barrier itself instead of waiting for a time-out of its own at the next one."""
import ctypes
import os
import subprocess

import pytest

from paper_1903_01665_gb300 import build as fgbuild

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
TIMEOUT_BIT = 1


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("team_barrier") / "team_barrier.so")
    subprocess.run([fgbuild._nvcc(), *fgbuild.ARCH, *fgbuild.NVCC_FLAGS, "-shared", "-cudart", "static",
                    os.path.join(HERE, "team_barrier.cu"), "-o", so], check=True)
    return ctypes.CDLL(so)


def _run(lib, grid, timeout_ms, late_ms):
    ok = (ctypes.c_int * grid)()
    took = (ctypes.c_uint64 * grid)()
    status = lib.run_late_arrival(grid, ctypes.c_double(timeout_ms), ctypes.c_double(late_ms), ok, took)
    return status, list(ok), [t / 1e6 for t in took]


@pytest.mark.parametrize("grid", [2, 7, 152])
def test_late_cta_learns_of_the_timeout(lib, grid):
    status, ok, took = _run(lib, grid, 40.0, 120.0)
    assert status == TIMEOUT_BIT and ok == [0] * grid
    assert all(t >= 39.0 for t in took[:-1])
    assert took[-1] < 20.0   # at once, not after a wait of its own


@pytest.mark.parametrize("grid", [2, 7, 152])
def test_late_cta_in_time(lib, grid):
    status, ok, _ = _run(lib, grid, 900.0, 20.0)
    assert status == 0 and ok == [1] * grid
