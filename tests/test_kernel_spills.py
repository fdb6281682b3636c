"""Orders that share only the call have kernels of their own: an order inlined beside another one takes registers from
graphs that never run it.  Reads what ptxas reports; the bounds are those before the orders were added."""
import os
import re
import subprocess

import pytest

from paper_1903_01665_gb300 import build as fgbuild

# fixpoint_kernel<algorithm, mode> -> largest spill stores, bytes
BOUNDS = {(0, 7): 96, (2, 10): 0, (2, 11): 0}   # near-far multi-source sweep; CC by hooking, 6 and 4 CTAs per SM


@pytest.fixture(scope="module")
def spills():
    src = os.path.join(fgbuild.CSRC, "fg_fixpoint.cu")
    out = subprocess.run([fgbuild._nvcc(), *fgbuild.ARCH, *fgbuild.NVCC_FLAGS, "-Xptxas", "-v", "-I",
                          os.path.join(fgbuild.ROOT, "include"), "-c", src, "-o", os.devnull],
                         check=True, capture_output=True, text=True).stderr
    found = re.findall(r"Function properties for \S*fixpoint_kernelILi(\d+)ELi(\d+)E\S*\n\s+\d+ bytes stack frame, "
                       r"(\d+) bytes spill stores", out)
    return {(int(a), int(m)): int(b) for a, m, b in found}


@pytest.mark.parametrize("kernel", list(BOUNDS))
def test_spills(spills, kernel):
    assert spills[kernel] <= BOUNDS[kernel]
