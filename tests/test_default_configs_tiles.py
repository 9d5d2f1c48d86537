"""The built-in choice where a plane is three tiles, so that a chunk of two and a
remainder both run: at each number of tiles where the choice changes and one
plane below it, y and dx equal those of candidate 0 bit for bit. The pixels are
small integers, so every FP32 partial sum is exact (16 tiles of at most 6 a
pixel stay below 2^24) and dw equals the FP64 sum: a tile left out or taken twice
shows."""
import pytest
import torch

from helpers import poison_like

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


def filter_gradient(x, dy, K):
    """The FP64 sums, 1024 planes at a time."""
    r, (H, W) = K // 2, x.shape[2:]
    dw = torch.zeros((K, K), dtype=torch.float64, device="cuda")
    for i in range(0, x.shape[0], 1024):
        xp = torch.nn.functional.pad(x[i:i + 1024].double(), (r, r, r, r))
        d = dy[i:i + 1024].double()
        for a in range(K):
            for b in range(K):
                dw[a, b] += (d * xp[:, :, a:a + H, b:b + W]).sum()
    return dw


@pytest.mark.parametrize("W", [128, 125])
@pytest.mark.parametrize("dtype,K,per_sm", [
    (torch.float32, 1, 80), (torch.float32, 3, 32), (torch.float32, 3, 100),
    (torch.float32, 9, 4), (torch.float32, 11, 4), (torch.float32, 11, 32),
    (torch.float32, 13, 4), (torch.float32, 15, 4), (torch.bfloat16, 1, 4),
    (torch.bfloat16, 3, 4), (torch.bfloat16, 5, 5), (torch.bfloat16, 7, 8),
    (torch.bfloat16, 9, 4), (torch.bfloat16, 11, 32), (torch.bfloat16, 15, 32)])
def test_three_tiles(giga, dtype, W, K, per_sm):
    from paper_2504_01266_gb300 import _lib as L
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    at = -(-per_sm * sms // 3)
    for planes in (at - 1, at):
        g = torch.Generator(device="cuda").manual_seed(K * planes + W)
        shape = (planes, 1, 129, W)
        x = torch.randint(0, 4, shape, generator=g, device="cuda").to(dtype)
        dy = torch.randint(-2, 3, shape, generator=g, device="cuda").to(dtype)
        w = torch.randn((1, K, K), generator=g, device="cuda") * 0.1
        d = L.desc(planes, 1, 1, 129, W, K, 1, L.GIGA_BORDER_ZERO, giga.DTYPES[dtype], 0)
        y = giga.conv2d_fwd(x, w, out=poison_like(x))
        dx, dw = giga.conv2d_bwd(x, dy, w, dx=poison_like(dy))
        for op in (1, 6):
            L.check(L.giga_autotune_set_choice(d, op, 0), "pin")
        assert torch.equal(y, giga.conv2d_fwd(x, w)), planes
        assert torch.equal(dx, giga.conv2d_bwd(x, dy, w)[0]), planes
        L.giga_autotune_clear()
        assert torch.equal(dw[0], filter_gradient(x, dy, K).float()), planes
