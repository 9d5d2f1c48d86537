"""The polyphase upsample's buffered rows (scales up to 8 that allow no wide
stores): widths around the 32 input columns of an item, each scale, both types
and borders, aligned and offset outputs, against the oracle; and the batched
plan equals the single call bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from helpers import BF16_KERNEL_TOL, assert_fp32, normwise, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def giga():
    import paper_2504_01266_gb300 as g
    from paper_2504_01266_gb300 import build
    build.build()
    return g


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("border", ["zero", "clamp"])
@pytest.mark.parametrize("scale,offset", [(2, 1), (3, 0), (3, 1), (4, 1), (5, 0), (6, 0), (7, 0),
                                          (7, 1), (8, 1), (9, 0)])
def test_widths_around_an_item(giga, dtype, border, scale, offset):
    b = oracle.ZERO if border == "zero" else oracle.CLAMP
    imgs = []
    for W in (1, 31, 32, 33, 65):
        gen = torch.Generator().manual_seed(100 * scale + W)
        x = torch.rand((1, 2, 9, W), generator=gen).to(dtype)
        w = torch.randn((2, 3, 3), generator=gen) * 0.1
        n = x.numel() * scale * scale
        buf = torch.full((n + 16,), float("nan"), dtype=dtype, device="cuda")
        y = buf[offset:offset + n].view(1, 2, 9 * scale, W * scale)
        giga.upsample_conv2d(x.cuda(), w.cuda(), scale, border, out=y)
        assert torch.isnan(buf[:offset]).all() and torch.isnan(buf[offset + n:]).all()
        xn, wn = x.float().numpy(), w.numpy()
        ref = oracle.upsample_dw_fwd(xn, wn, b, scale)
        if dtype == torch.float32:
            mag = oracle.upsample_dw_fwd(np.abs(xn), np.abs(wn), b, scale)
            assert_fp32(to_np(y), ref, mag, 13, (scale, W))  # 9 tap sums and 4 multiply-adds
        else:
            assert normwise(to_np(y), ref) <= BF16_KERNEL_TOL
        batch_y = torch.full_like(buf, float("nan"))[offset:offset + n].view(y.shape)[0]
        imgs.append((dict(x=x.cuda()[0], w=w.cuda(), scale=scale, y=batch_y), y))
    plan = giga.UpsampleBatchedPlan([im for im, _ in imgs], border, dtype)
    plan.upload()
    plan.run()
    for im, y in imgs:
        assert torch.equal(im["y"], y[0])
    plan.close()
