"""The filter gradient of BF16 planes that TMA cannot load, on both sides of the
tile counts and sizes where its warps' layout changes: against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from helpers import assert_fp32, to_np
from test_row_alignment import at_offset

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def giga():
    import paper_2504_01266_gb300 as g
    from paper_2504_01266_gb300 import build
    build.build()
    return g


@pytest.mark.parametrize("K", [1, 3, 5, 7, 13])
@pytest.mark.parametrize("H,W,offset,extra", [(65, 127, 0, 0), (65, 127, 0, 1), (64, 125, 0, 0),
                                              (65, 126, 0, 0), (65, 128, 4, 0), (3, 131, 0, 1)])
def test_bf16(giga, K, H, W, offset, extra):
    """Planes of two tiles (one: 64 x 125), in all 6 tiles per SM or just more."""
    tpp = -(-H // 64) * -(-W // 128)
    planes = 6 * torch.cuda.get_device_properties(0).multi_processor_count // tpp + extra
    border = oracle.CLAMP if K % 4 == 1 else oracle.ZERO
    gen = torch.Generator().manual_seed(K + W)
    x = torch.rand((planes, 1, H, W), generator=gen).bfloat16()
    dy = torch.randn((planes, 1, H, W), generator=gen).bfloat16()
    dw = giga.conv2d_bwd_filter(at_offset(x, offset)[0], at_offset(dy, offset)[0], K,
                                "clamp" if border == oracle.CLAMP else "zero")
    xn, dyn = x.float().numpy(), dy.float().numpy()
    assert_fp32(to_np(dw), oracle.dw_bwd_filter(xn, dyn, K, border),
                oracle.dw_bwd_filter(np.abs(xn), np.abs(dyn), K, border), planes * H * W, (K, W))
