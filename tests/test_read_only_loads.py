"""Data that a kernel writes is not read through the read-only path: the
element load the kernels use does not compile for a pointer to non-const
data (the edge fold read the input gradient it writes that way)."""
import os
import subprocess

import pytest

from paper_2504_01266_gb300 import build

SOURCE = """
#include "common.cuh"
__global__ void copy(%s* p, float* out) { *out = giga::Elem<%s>::load(p); }
"""


@pytest.mark.parametrize("elem", ["float", "__nv_bfloat16"])
def test_load_takes_const_data_only(tmp_path, elem):
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    codes = []
    for qual in ("const ", ""):
        src = tmp_path / "load.cu"
        src.write_text(SOURCE % (qual + elem, elem))
        codes.append(subprocess.run([nvcc, *build.ARCH, *build.NVCC_FLAGS, "-c", str(src), "-o",
                                     os.devnull], capture_output=True, timeout=300).returncode)
    assert codes[0] == 0 and codes[1] != 0, codes
