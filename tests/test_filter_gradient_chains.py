"""How many terms of a filter gradient are added one after the other in FP32
before FP64 (or a sum of few) takes over.  One pixel of dy is 1 and others are
2^-25, which FP32 cannot add to 1 one by one but keeps when they meet first;
x = 1, so the centre tap's gradient is their sum."""
import pytest
import torch

pytestmark = pytest.mark.gpu

SMALL = 2.0 ** -25


@pytest.fixture(scope="module")
def giga():
    import paper_2504_01266_gb300 as g
    from paper_2504_01266_gb300 import _lib, build
    build.build()
    mode = _lib.giga_autotune_get_mode()
    _lib.giga_autotune_clear()
    _lib.giga_autotune_set_mode(1)
    yield g
    _lib.giga_autotune_clear()
    _lib.giga_autotune_set_mode(mode)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("W", [128, 125])
@pytest.mark.parametrize("K,rows", [(1, 8), (3, 8), (5, 8), (7, 8), (11, 16)])
def test_filter_kernel_rows(giga, dtype, W, K, rows):
    """The rows x 4 pixels of a lane: half of them do not follow the 1."""
    dy = torch.zeros((1, 1, 64, W), dtype=dtype, device="cuda")
    dy[0, 0, :rows, 64:68] = SMALL
    dy[0, 0, 0, 64] = 1.0
    dw = giga.conv2d_bwd_filter(torch.ones_like(dy), dy, K)
    assert dw[0, K // 2, K // 2].item() >= 1.0 + 2 * rows * SMALL


@pytest.mark.parametrize("dtype,K,per_sm,tile", [
    (torch.float32, 3, 16, 1), (torch.float32, 3, 40, 1), (torch.bfloat16, 1, 4, 1),
    (torch.bfloat16, 3, 4, 1),
    (torch.float32, 9, 4, 2), (torch.float32, 11, 4, 4), (torch.bfloat16, 7, 8, 2),
    (torch.float32, 13, 4, 4)])
def test_both_gradients_tiles(giga, dtype, K, per_sm, tile):
    """Both gradients from the tile count on where the built-in choice leaves the
    fused kernel (which takes one tile per partial sum there): the pixels of the
    tiles from `tile` on do not follow the 1 of the first."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    planes = per_sm * sms // 8 + 1  # of eight tiles each
    dy = torch.zeros((planes, 1, 512, 128), dtype=dtype, device="cuda")
    for t in range(tile, 8):
        dy[0, 0, 64 * t:64 * t + 4, 64:68] = SMALL
    dy[0, 0, 0, 64] = 1.0
    w = torch.zeros((1, K, K), device="cuda")
    dw = giga.conv2d_bwd(torch.ones_like(dy), dy, w)[1]
    assert dw[0, K // 2, K // 2].item() == 1.0 + 16 * (8 - tile) * SMALL
