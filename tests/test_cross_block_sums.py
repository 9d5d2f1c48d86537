"""The sums across blocks of the filter gradients (two-float sums closed in
FP64): infinities and NaN come through, partial sums that overflow FP32 on the
way to a finite total do not spoil it, and cancelling partials keep the digits
FP64 keeps."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def giga():
    import paper_2504_01266_gb300 as g
    from paper_2504_01266_gb300 import build
    build.build()
    return g


def single_pixels(values):
    """One value per 64-row tile (so per chunk of one tile) of a 128-wide plane,
    x = 1: the centre tap's gradient is their sum."""
    dy = torch.zeros((1, 1, 64 * len(values), 128))
    for i, v in enumerate(values):
        dy[0, 0, 64 * i + 32, 64] = v
    return torch.ones_like(dy).cuda(), dy.cuda()


CASES = [([3e38, 3e38, -3e38, -3e38, 2.0 ** 100], 2.0 ** 100),  # overflows FP32 in order
         ([1.0, 2.0 ** 30, 2.0 ** -20, -(2.0 ** 30)], 1.0 + 2.0 ** -20),
         ([1.0, float("inf"), 2.0], float("inf")),
         ([float("inf"), -float("inf")], float("nan")),
         ([1.0, float("nan"), 2.0], float("nan"))]


@pytest.mark.parametrize("values,total", CASES)
def test_depthwise_and_ragged(giga, values, total):
    K = 3
    x, dy = single_pixels(values)
    w = torch.zeros((1, K, K)).cuda()
    got = [giga.conv2d_bwd_filter(x, dy, K)[0, 1, 1].item(),
           giga.conv2d_bwd(x, dy, w)[1][0, 1, 1].item()]
    if not np.isfinite(total):  # the plan's chunks of four tiles sum these in FP32
        dw = torch.empty_like(w)
        plan = giga.BatchedPlan([dict(x=x[0], dy=dy[0], w=w, dw=dw)], 4)
        plan.upload()
        plan.run()
        got.append(dw[0, 1, 1].item())
        plan.close()
    for v in got:
        np.testing.assert_equal(np.float32(v), np.float32(total))


def test_dense_non_finite(giga):
    x = torch.ones((1, 40, 300, 64), dtype=torch.bfloat16).cuda()
    dy = torch.zeros_like(x)
    dy[0, 20, 100, 3] = float("inf")
    dy[0, 5, 200, 7] = float("nan")
    dw = giga.dense_conv2d_bwd_filter(x, dy)
    assert torch.isinf(dw[3]).all() and torch.isnan(dw[7]).all()
    rest = torch.ones(64, dtype=torch.bool)
    rest[[3, 7]] = False
    assert (dw[rest.cuda()] == 0).all()
