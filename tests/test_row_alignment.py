"""Rows at every alignment: image widths of every residue modulo 16 bytes and
tensors that start at any element of a larger buffer, for each depthwise entry
point that stages rows without TMA.  Widths just above three 128-column tiles
give left, inner and right tiles; the inputs sit in a buffer of NaNs (a read
outside the rows would show) and so do the outputs (a write outside would
show, and so would a pixel that is not written)."""
import numpy as np
import pytest
import torch

import oracle
from helpers import BF16_KERNEL_TOL, FP32_TOL, assert_fp32, normwise, to_np

pytestmark = pytest.mark.gpu

BORDER = {"zero": oracle.ZERO, "clamp": oracle.CLAMP}


@pytest.fixture(scope="module")
def giga():
    import paper_2504_01266_gb300 as g
    from paper_2504_01266_gb300 import build
    build.build()
    return g


def at_offset(t, offset):
    """t on the device, `offset` elements into a buffer of NaNs; and that buffer."""
    buf = torch.full((t.numel() + offset + 16,), float("nan"), dtype=t.dtype, device="cuda")
    v = buf[offset:offset + t.numel()].view(t.shape)
    v.copy_(t)
    return v, buf


def hole(shape, dtype, offset):
    return at_offset(torch.full(shape, float("nan"), dtype=dtype), offset)


def untouched(buf, offset, n):
    return bool(torch.isnan(buf[:offset]).all() and torch.isnan(buf[offset + n:]).all())


CASES = [(W, off) for W in range(385, 393) for off in (0, 1)] + [(388, 2), (388, 3), (390, 5),
                                                                 (392, 4), (130, 1), (5, 3)]


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("K", [1, 3, 7, 15])
@pytest.mark.parametrize("W,offset", CASES)
def test_forward_and_gradients(giga, dtype, K, W, offset):
    border = "clamp" if (W + offset) % 2 else "zero"
    shape, b = (1, 2, 70, W), BORDER[border]
    gen = torch.Generator().manual_seed(1000 * K + 10 * W + offset)
    x, dy = torch.rand(shape, generator=gen).to(dtype), torch.randn(shape, generator=gen).to(dtype)
    w = torch.randn((2, K, K), generator=gen) * 0.1
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
    rdw = oracle.dw_bwd_filter(xn, dyn, K, b)
    what = (W, offset, K, border)
    if dtype == torch.float32:
        assert_fp32(to_np(y), ry, oracle.dw_fwd(ax, aw, b), K * K, what)
        assert_fp32(to_np(dx), rdx, oracle.dw_bwd_input(ady, aw, b),
                    (K // 2 + 1) ** 2 * K * K, what)
    else:
        assert normwise(to_np(y), ry) <= BF16_KERNEL_TOL, what
        assert normwise(to_np(dx), rdx) <= BF16_KERNEL_TOL, what
    mag = oracle.dw_bwd_filter(ax, ady, K, b)
    assert_fp32(to_np(dw), rdw, mag, 70 * W, what)
    assert_fp32(to_np(dw_only), rdw, mag, 70 * W, what)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("W,offset", CASES)
def test_separable_gray_and_wide_filters(giga, dtype, W, offset):
    border = "zero" if (W + offset) % 2 else "clamp"
    b = BORDER[border]
    gen = torch.Generator().manual_seed(77 * W + offset)
    x = torch.rand((1, 3, 70, W), generator=gen).to(dtype)
    xc, xn = at_offset(x, offset)[0], x.float().numpy()
    tol = FP32_TOL if dtype == torch.float32 else BF16_KERNEL_TOL
    for K in (3, 9, 15):
        f = torch.rand((3, K), generator=gen) / K
        y, buf = hole(x.shape, dtype, offset)
        giga.conv2d_separable(xc, f.cuda(), f.cuda(), border, out=y)
        full = (f.double()[:, :, None] * f.double()[:, None, :]).numpy()
        assert untouched(buf, offset, x.numel())
        assert normwise(to_np(y), oracle.dw_fwd(xn.astype(np.float64), full, b)) <= tol, (W, K)
    for K in (17, 31):
        w = torch.rand((3, K, K), generator=gen) / (K * K)
        y, buf = hole(x.shape, dtype, offset)
        giga.conv2d_fwd(xc, w.cuda(), border, out=y)
        assert untouched(buf, offset, x.numel())
        assert normwise(to_np(y), oracle.dw_fwd(xn, w.numpy(), b)) <= tol, (W, K)
    for K in (3, 7):
        w = torch.rand((1, K, K), generator=gen) / (K * K)
        y, buf = hole((1, 1, 70, W), dtype, offset)
        giga.gray_conv2d(xc, w.cuda(), border, out=y)
        gray = oracle.rgb_to_gray(xn)
        assert untouched(buf, offset, 70 * W)
        assert normwise(to_np(y), oracle.dw_fwd(gray, w.numpy().astype(np.float64), b)) <= tol


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("border", ["zero", "clamp"])
def test_ragged_batch(giga, dtype, border):
    """One batch with every width and offset equals the per-image calls bit for
    bit (y, dx) and their filter gradients within the FP32 bound."""
    gen = torch.Generator().manual_seed(9)
    imgs, refs = [], []
    for i, (W, offset) in enumerate(CASES):
        K = (1, 3, 5, 7, 9, 11, 13, 15)[i % 8]
        x, dy = torch.rand((2, 70, W), generator=gen), torch.randn((2, 70, W), generator=gen)
        w = (torch.randn((2, K, K), generator=gen) * 0.1).cuda()
        xc, dyc = at_offset(x.to(dtype), offset)[0], at_offset(dy.to(dtype), offset)[0]
        y, dx = hole(x.shape, dtype, offset), hole(x.shape, dtype, offset)
        imgs.append(dict(x=xc, dy=dyc, w=w, y=y[0], dx=dx[0], dw=torch.empty_like(w)))
        refs.append((offset, y[1], dx[1]))
    plan = giga.BatchedPlan(imgs, 7, border, dtype=dtype)
    plan.upload()
    plan.run()
    for im, (offset, ybuf, dxbuf) in zip(imgs, refs):
        n = im["x"].numel()
        assert untouched(ybuf, offset, n) and untouched(dxbuf, offset, n)
        y = giga.conv2d_fwd(im["x"][None], im["w"], border)[0]
        dx, dw = giga.conv2d_bwd(im["x"][None], im["dy"][None], im["w"], border)
        assert torch.equal(im["y"], y)
        if border == "zero":  # the clamp fold adds in another order
            assert torch.equal(im["dx"], dx[0])
        else:
            assert normwise(to_np(im["dx"]), to_np(dx[0])) <= (
                FP32_TOL if dtype == torch.float32 else BF16_KERNEL_TOL)
        assert normwise(to_np(im["dw"]), to_np(dw)) <= FP32_TOL
    plan.close()
