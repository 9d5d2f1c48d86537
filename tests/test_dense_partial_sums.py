"""The dense filter gradient's sums over blocks: exact where FP64's are (values of
8 bits over 2^30 of range, one per block), and finite totals of partial sums that
overflow FP32 on the way."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def giga():
    import paper_2504_01266_gb300 as g
    from paper_2504_01266_gb300 import build
    build.build()
    return g


def gradient(giga, rows):
    """dw's centre taps for one value per block and output channel: rows is
    (blocks, 64); every block has one row of one 62-pixel-wide image."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    x = torch.ones((1, sms, 62, 64), dtype=torch.bfloat16, device="cuda")
    dy = torch.zeros_like(x)
    dy[0, :, 30] = rows.to(dy)
    dw = giga.dense_conv2d_bwd_filter(x, dy)[:, 1, 1]
    assert (dw == dw[:, :1]).all()  # every input channel has x = 1
    return dw[:, 0].cpu()


def test_exact(giga):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    gen = torch.Generator().manual_seed(5)
    scale = 2.0 ** torch.randint(-15, 16, (sms, 64), generator=gen).float()
    rows = (torch.randn((sms, 64), generator=gen) * scale).bfloat16().float()
    rows[sms // 2:sms // 2 * 2] = -rows[:sms // 2].roll(3, 0)  # cancel, across the groups
    rows[:, 1::2] += 2.0 ** -8  # a rest that FP32 sums lose
    rows = rows.bfloat16().float()
    want = torch.tensor([math.fsum(rows[:, o].tolist()) for o in range(64)], dtype=torch.float64)
    assert torch.equal(gradient(giga, rows), want.float())


def test_overflow_on_the_way(giga):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = torch.zeros((sms, 64))
    for i, v in enumerate([3e38, 3e38, -3e38, -3e38, 2.0 ** 100]):
        rows[20 + 4 * i] = v
    assert (gradient(giga, rows) == 2.0 ** 100).all()
