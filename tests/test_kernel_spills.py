"""Orders that share only the call have kernels of their own: an order inlined beside another one takes registers from
graphs that never run it.  Reads what ptxas reports; the bounds are those before the orders were added."""
import os
import re
import subprocess

import pytest

from paper_1903_01665_gb300 import build as fgbuild

# kernel -> largest spill stores, bytes: the near-far multi-source sweep; CC by hooking with 6 and 4 CTAs per SM; the
# all-active vertex sweep of graphs that fill its warps
BOUNDS = {"fixpoint_kernelILi0ELi7E": 96, "fixpoint_kernelILi2ELi10E": 0, "fixpoint_kernelILi2ELi11E": 0,
          "sweep_kernelILi0ELb0E": 0}


@pytest.fixture(scope="module")
def spills():
    src = os.path.join(fgbuild.CSRC, "fg_fixpoint.cu")
    out = subprocess.run([fgbuild._nvcc(), *fgbuild.ARCH, *fgbuild.NVCC_FLAGS, "-Xptxas", "-v", "-I",
                          os.path.join(fgbuild.ROOT, "include"), "-c", src, "-o", os.devnull],
                         check=True, capture_output=True, text=True).stderr
    found = re.findall(r"Function properties for \S*?((?:fixpoint|sweep)_kernelI(?:L[ib]\d+E)+)\S*\n"
                       r"\s+\d+ bytes stack frame, (\d+) bytes spill stores", out)
    return {k: int(b) for k, b in found}


@pytest.mark.parametrize("kernel", list(BOUNDS))
def test_spills(spills, kernel):
    assert spills[kernel] <= BOUNDS[kernel]
