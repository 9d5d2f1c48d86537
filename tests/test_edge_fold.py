"""The clamp-border edge fold and the filter-gradient sums that follow the
backward tile passes in one launch: planes one and two pixels high or wide
(where an edge pixel lies on several edges), edges just below, at and above the
256 pixels of a fold block, filters larger than the image, and channel counts
that take every number of taps per block."""
import numpy as np
import pytest
import torch

import oracle
from helpers import assert_fp32, poison_like, to_np

pytestmark = pytest.mark.gpu

SHAPES = [(1, 2, 1, 1), (1, 2, 1, 300), (1, 2, 300, 1), (2, 1, 2, 2), (1, 1, 2, 257),
          (1, 1, 257, 2), (1, 2, 3, 256), (2, 1, 258, 255), (1, 1, 6, 9)]


@pytest.fixture(scope="module")
def giga():
    import paper_2504_01266_gb300 as g
    from paper_2504_01266_gb300 import build
    build.build()
    return g


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("K", [3, 5, 15, 31])
@pytest.mark.parametrize("shape", SHAPES)
def test_input_gradient_clamp(giga, dtype, K, shape):
    gen = torch.Generator().manual_seed(31 * K + shape[2] + 7 * shape[3])
    dy = torch.randn(shape, generator=gen).to(dtype)
    w = torch.randn((shape[1], K, K), generator=gen) * 0.1
    dx = giga.conv2d_bwd_input(dy.cuda(), w.cuda(), "clamp", out=poison_like(dy.cuda()))
    dyn, wn = dy.float().numpy(), w.numpy()
    ref = oracle.dw_bwd_input(dyn, wn, oracle.CLAMP)
    mag = oracle.dw_bwd_input(np.abs(dyn), np.abs(wn), oracle.CLAMP)
    if dtype == torch.float32:
        # an edge pixel sums up to (r + 1)^2 K^2 terms, and more where it lies on
        # opposite edges: at most every pixel's K^2
        n = max((K // 2 + 1) ** 2, min(shape[2], K) * min(shape[3], K)) * K * K
        assert_fp32(to_np(dx), ref, mag, n, (shape, K))
    else:
        out = to_np(dx)
        # FP32 sums of those terms (2^-13 of their magnitudes at most), one rounding to storage
        assert not np.isnan(out).any()
        assert (np.abs(out - ref) <= 2.0 ** -8 * np.abs(ref) + 2.0 ** -13 * mag).all()


@pytest.mark.parametrize("C,K", [(1, 1), (3, 3), (40, 3), (5, 15), (64, 5), (130, 7)])
@pytest.mark.parametrize("N", [1, 5])
def test_filter_gradient_sums(giga, C, K, N):
    """Both gradients; the sums over many channels take 1 to 32 taps per block."""
    gen = torch.Generator().manual_seed(C * K + N)
    shape = (N, C, 70, 140)
    x, dy = torch.rand(shape, generator=gen), torch.randn(shape, generator=gen)
    w = torch.randn((C, K, K), generator=gen) * 0.1
    xc, dyc = x.cuda(), dy.cuda()
    dx, dw = giga.conv2d_bwd(xc, dyc, w.cuda(), "clamp", dx=poison_like(dyc))
    again = giga.conv2d_bwd(xc, dyc, w.cuda(), "clamp")[1]
    assert torch.equal(dw, again)  # a fixed order
    xn, dyn, wn = x.numpy(), dy.numpy(), w.numpy()
    assert_fp32(to_np(dw), oracle.dw_bwd_filter(xn, dyn, K, oracle.CLAMP),
                oracle.dw_bwd_filter(np.abs(xn), np.abs(dyn), K, oracle.CLAMP), N * 70 * 140, "dw")
    assert_fp32(to_np(dx), oracle.dw_bwd_input(dyn, wn, oracle.CLAMP),
                oracle.dw_bwd_input(np.abs(dyn), np.abs(wn), oracle.CLAMP),
                (K // 2 + 1) ** 2 * K * K, "dx")
