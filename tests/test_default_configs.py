"""The configurations a call takes when the tuner holds no choice (by filter
size, type, alignment and tile count): at, just below and just above each
number of tiles where the rule changes, y and dx equal those of candidate 0
bit for bit (the order of a pixel's sum does not depend on the configuration)
and dw agrees within the FP32 bound."""
import pytest
import torch

from helpers import assert_fp32, poison_like, to_np

pytestmark = pytest.mark.gpu


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
@pytest.mark.parametrize("K,per_sm", [(1, 16), (1, 80), (3, 2), (3, 4), (3, 16), (3, 100), (5, 8),
                                      (7, 8), (7, 16), (9, 4), (11, 4), (11, 16), (13, 2), (15, 2)])
def test_both_sides_of_each_threshold(giga, dtype, W, K, per_sm):
    from paper_2504_01266_gb300 import _lib as L
    H = 33 if per_sm <= 16 else 3  # the bound needs planes * H * W below 2^24
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for planes in (per_sm * sms - 1, per_sm * sms, per_sm * sms + 1):  # one tile each
        g = torch.Generator(device="cuda").manual_seed(K * planes)
        shape = (planes, 1, H, W)
        x = torch.rand(shape, generator=g, device="cuda").to(dtype)
        dy = torch.randn(shape, generator=g, device="cuda").to(dtype)
        w = torch.randn((1, K, K), generator=g, device="cuda") * 0.1
        d = L.desc(planes, 1, 1, H, W, K, 1, L.GIGA_BORDER_ZERO, giga.DTYPES[dtype], 0)
        got = []
        for pinned in (False, True):
            if pinned:
                for op in (1, 2, 4, 6):
                    L.check(L.giga_autotune_set_choice(d, op, 0), "pin")
            y = giga.conv2d_fwd(x, w, out=poison_like(x))
            dx1 = giga.conv2d_bwd_input(dy, w, out=poison_like(dy))
            dx2, dw = giga.conv2d_bwd(x, dy, w, dx=poison_like(dy))
            got.append((y, dx1, dx2, dw))
        L.giga_autotune_clear()
        (y, dx1, dx2, dw), (y0, dx10, dx20, dw0) = got
        assert torch.equal(y, y0) and torch.equal(dx1, dx10), (planes, K)
        assert torch.equal(dx2, dx20) and torch.equal(dx1, dx2), (planes, K)
        mag = giga.conv2d_bwd(x.abs(), dy.abs(), w)[1]
        assert_fp32(to_np(dw), to_np(dw0), 2 * to_np(mag), planes * H * W, (planes, K))
