"""The one-step kernels are dependent launches (launch_pdl): they live while
the kernel before them still writes, so none of their loads may take the
read-only path, which is for data that nothing writes meanwhile.  Checked in
the sources: neither the intrinsic nor pointers that let the compiler choose
that path.  (The fused batch is an ordinary launch.)"""
import os
import re

import pytest

from paper_2112_13169_gb300 import build

FILES = sorted(f for f in os.listdir(build.CSRC) if f.endswith((".cu", ".cuh")) and f != "k_batch.cu")


@pytest.mark.parametrize("name", FILES)
def test_dependent_launches_take_no_read_only_loads(name):
    src = open(os.path.join(build.CSRC, name)).read()
    code = re.sub(r"//[^\n]*|/\*.*?\*/", "", src, flags=re.S)
    for bad in ("__ldg", "LoadRO", "global.nc", "__restrict"):
        assert bad not in code, "%s: %s" % (name, bad)


def test_the_fused_batch_is_no_dependent_launch():
    src = open(os.path.join(build.CSRC, "k_batch.cu")).read()
    assert "cudaLaunchCooperativeKernel" in src and "launch_pdl" not in src
