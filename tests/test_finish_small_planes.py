"""What follows the backward tile passes on small planes and few partial sums:
edges around the 64 pixels of a small fold block and the 128 where the large
ones begin, many channels of planes smaller than the filter (the last shape has
more than four planes per SM, where BF16 goes pixel by pixel for K <= 5), and
channel counts (from the device's SM count) that take each number of taps per
block."""
import numpy as np
import pytest
import torch

import oracle
from helpers import assert_fp32, poison_like, to_np

pytestmark = pytest.mark.gpu

SHAPES = [(1, 2, 63, 65), (2, 1, 64, 128), (1, 2, 128, 127), (1, 1, 129, 64), (1, 1, 2, 128),
          (2, 70, 7, 7), (3, 40, 14, 5), (5, 130, 7, 6)]


@pytest.fixture(scope="module")
def giga():
    import paper_2504_01266_gb300 as g
    from paper_2504_01266_gb300 import build
    build.build()
    return g


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("K", [3, 5, 15, 31])
@pytest.mark.parametrize("shape", SHAPES)
def test_edge_fold(giga, dtype, K, shape):
    gen = torch.Generator().manual_seed(37 * K + shape[2] + 11 * shape[3])
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
        assert not np.isnan(out).any()
        # FP32 sums of those terms (2^-13 of their magnitudes at most), one rounding to storage
        assert (np.abs(out - ref) <= 2.0 ** -8 * np.abs(ref) + 2.0 ** -13 * mag).all()


@pytest.mark.parametrize("taps", [1, 2, 4, 8, 16, 32])
@pytest.mark.parametrize("N", [1, 3, 40])
def test_taps_per_block(giga, taps, N):
    """The most channels for which `taps` taps per block give at most two blocks
    per SM (fewer taps would give more)."""
    K = 7
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    C = 2 * sms // ((K * K + taps - 1) // taps)
    gen = torch.Generator().manual_seed(C + N)
    shape = (N, C, 9, 12)
    x, dy = torch.rand(shape, generator=gen), torch.randn(shape, generator=gen)
    w = torch.randn((C, K, K), generator=gen) * 0.1
    xc, dyc = x.cuda(), dy.cuda()
    dx, dw = giga.conv2d_bwd(xc, dyc, w.cuda(), "clamp", dx=poison_like(dyc))
    dw_only = giga.conv2d_bwd_filter(xc, dyc, K, "clamp")
    xn, dyn, wn = x.numpy(), dy.numpy(), w.numpy()
    ref = oracle.dw_bwd_filter(xn, dyn, K, oracle.CLAMP)
    mag = oracle.dw_bwd_filter(np.abs(xn), np.abs(dyn), K, oracle.CLAMP)
    for d in (dw, dw_only):
        assert_fp32(to_np(d), ref, mag, N * 9 * 12, "dw")
    assert_fp32(to_np(dx), oracle.dw_bwd_input(dyn, wn, oracle.CLAMP),
                oracle.dw_bwd_input(np.abs(dyn), np.abs(wn), oracle.CLAMP),
                (K // 2 + 1) ** 2 * K * K, "dx")
