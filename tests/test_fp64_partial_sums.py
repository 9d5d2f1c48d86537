"""The filter gradients' sums across blocks keep FP64's 53 bits: partial sums
whose exact total survives the cancellation of terms 2^26 and 1 around it.
Every subset of the five values is exact in FP64, so the total is, in any order
of the FP64 sum; sums with fewer bits lose it.  The values lie as many partial
sums apart as one thread steps, so that one thread meets all of them."""
import pytest
import torch

pytestmark = pytest.mark.gpu

VALUES = [2.0 ** 26, 1.0, 2.0 ** -25, -1.0, -(2.0 ** 26)]
TOTAL = 2.0 ** -25


@pytest.fixture(scope="module")
def giga():
    import paper_2504_01266_gb300 as g
    from paper_2504_01266_gb300 import build
    build.build()
    return g


@pytest.mark.parametrize("stride", [1, 16, 128, 512])
def test_depthwise(giga, stride):
    """One partial sum per image; a thread adds those of every 512th image."""
    dy = torch.zeros((4 * stride + 1, 1, 1, 128), device="cuda")
    for i, v in enumerate(VALUES):
        dy[i * stride, 0, 0, 64] = v
    x, w = torch.ones_like(dy), torch.zeros((1, 3, 3), device="cuda")
    for dw in (giga.conv2d_bwd_filter(x, dy, 3), giga.conv2d_bwd(x, dy, w)[1]):
        assert (dw[0, 1] == TOTAL).all()


@pytest.mark.parametrize("stride", [1, 16])
def test_ragged(giga, stride):
    """One value per chunk of the plan's four tiles of 64 rows; a thread adds
    the partial sums of every 16th chunk."""
    dy = torch.zeros((1, 256 * (4 * stride + 1), 128), device="cuda")
    for i, v in enumerate(VALUES):
        dy[0, 256 * i * stride + 32, 64] = v
    x, dw = torch.ones_like(dy), torch.empty((1, 3, 3), device="cuda")
    plan = giga.BatchedPlan([dict(x=x, dy=dy, dw=dw)], 4)
    assert plan.tiles_per_chunk == 4
    plan.upload()
    plan.run()
    torch.cuda.synchronize()
    plan.close()
    assert (dw == TOTAL).all()


def test_dense(giga):
    """One row of one 62-pixel-wide image per block; a thread adds the partial
    sums of every fourth block."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    x = torch.ones((1, sms, 62, 64), dtype=torch.bfloat16, device="cuda")
    dy = torch.zeros_like(x)
    for i, v in enumerate(VALUES):
        dy[0, 20 + 4 * i, 30, ::3] = v
    dw = giga.dense_conv2d_bwd_filter(x, dy)
    assert (dw[::3] == TOTAL).all()
    rest = torch.ones(64, dtype=torch.bool)
    rest[::3] = False
    assert (dw[rest.cuda()] == 0).all()
