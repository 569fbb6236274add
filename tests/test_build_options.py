"""The compile-time options of csrc/decide.cuh: the kernels that lay out tables by
them compile for either width of tier 2 (needs nvcc, no GPU)."""
import os
import subprocess

import pytest

from paper_2608_03695_gb300 import build_lib


@pytest.mark.parametrize("lanes", [16, 32])
def test_tier2_lanes(lanes, tmp_path):
    if not os.path.exists(build_lib.NVCC):
        pytest.skip("no nvcc")
    src = tmp_path / "options.cu"
    src.write_text('#include "resident.cuh"\n')
    r = subprocess.run([build_lib.NVCC, *build_lib.ARCH, *build_lib.FLAGS, f"-DMSLICE_T2_LANES={lanes}", "-I",
                        build_lib.CSRC, "-c", str(src), "-o", str(tmp_path / "options.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
