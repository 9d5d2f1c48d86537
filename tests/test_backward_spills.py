"""The fused backward kernels of the sizes where registers are tight keep (next to)
nothing in local memory: what ptxas reports for them."""
import concurrent.futures
import re

import pytest

from paper_2504_01266_gb300 import build


def spilled(K):
    """Bytes of spill stores of each fused backward kernel of filter size K."""
    report = build.ptxas_report(f"dw_k{K:02d}.cu")
    found = re.findall(r"Function properties for (\S*\d+dw_bwd_kernel\S*)\s+\d+ bytes stack frame, "
                       r"(\d+) bytes spill stores", report)
    return {name: int(n) for name, n in found}


def test_spills():
    try:
        build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    with concurrent.futures.ThreadPoolExecutor(4) as pool:
        sizes = dict(zip((5, 11, 13, 15), pool.map(spilled, (5, 11, 13, 15))))
    for K, kernels in sizes.items():
        assert len(kernels) == 6, (K, kernels)  # two types, three alignments
        assert all(n <= 32 for n in kernels.values()), (K, kernels)
