"""Images much smaller than a tile, at every alignment: heights on both sides of
half a tile, inputs and outputs framed by NaNs (a read or a write outside
would show), all depthwise passes against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from helpers import BF16_KERNEL_TOL, assert_fp32, normwise, to_np
from test_row_alignment import BORDER, at_offset, hole, untouched

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def giga():
    import paper_2504_01266_gb300 as g
    from paper_2504_01266_gb300 import build
    build.build()
    return g


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("K", [1, 3, 11])
@pytest.mark.parametrize("H", [1, 7, 16, 17, 31, 33, 38])
@pytest.mark.parametrize("W,offset", [(7, 0), (14, 1), (129, 0), (250, 3)])
def test_all_passes(giga, dtype, K, H, W, offset):
    border = "clamp" if (H + W) % 2 else "zero"
    shape, b = (2, 3, H, W), BORDER[border]
    gen = torch.Generator().manual_seed(1000 * K + 10 * W + H)
    x, dy = torch.rand(shape, generator=gen).to(dtype), torch.randn(shape, generator=gen).to(dtype)
    w = torch.randn((3, K, K), generator=gen) * 0.1
    xc, dyc, wc = at_offset(x, offset)[0], at_offset(dy, offset)[0], w.cuda()
    y, ybuf = hole(shape, dtype, offset)
    giga.conv2d_fwd(xc, wc, border, out=y)
    dx, dxbuf = hole(shape, dtype, offset)
    _, dw = giga.conv2d_bwd(xc, dyc, wc, border, dx=dx)
    dw_only = giga.conv2d_bwd_filter(xc, dyc, K, border)
    n = x.numel()
    assert untouched(ybuf, offset, n) and untouched(dxbuf, offset, n)
    xn, dyn, wn = x.float().numpy(), dy.float().numpy(), w.numpy()
    ax, ady, aw = np.abs(xn), np.abs(dyn), np.abs(wn)
    ry, rdx = oracle.dw_fwd(xn, wn, b), oracle.dw_bwd_input(dyn, wn, b)
    what, terms = (H, W, K, border), max((K // 2 + 1) ** 2, min(H, K) * min(W, K)) * K * K
    if dtype == torch.float32:
        assert_fp32(to_np(y), ry, oracle.dw_fwd(ax, aw, b), K * K, what)
        assert_fp32(to_np(dx), rdx, oracle.dw_bwd_input(ady, aw, b), terms, what)
    else:
        assert normwise(to_np(y), ry) <= BF16_KERNEL_TOL, what
        assert normwise(to_np(dx), rdx) <= BF16_KERNEL_TOL, what
    rdw = oracle.dw_bwd_filter(xn, dyn, K, b)
    mag = oracle.dw_bwd_filter(ax, ady, K, b)
    assert_fp32(to_np(dw), rdw, mag, 2 * H * W, what)
    assert_fp32(to_np(dw_only), rdw, mag, 2 * H * W, what)
