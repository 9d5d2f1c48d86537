"""Inputs that TMA can load with outputs at any element of a larger buffer (NaNs
around them): the same results, bit for bit, as with aligned outputs."""
import pytest
import torch

from test_row_alignment import hole, untouched

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
@pytest.mark.parametrize("K", [1, 3, 5, 7, 9, 11, 13, 15])
@pytest.mark.parametrize("W,offset", [(8, 1), (128, 1), (136, 3), (392, 2)])
def test_depthwise(giga, dtype, K, W, offset):
    from paper_2504_01266_gb300 import _lib as L
    border = "clamp" if (K + offset) % 4 else "zero"
    shape = (2, 3, 70, W)
    g = torch.Generator(device="cuda").manual_seed(100 * K + W)
    x = torch.rand(shape, generator=g, device="cuda").to(dtype)
    dy = torch.randn(shape, generator=g, device="cuda").to(dtype)
    w = torch.randn((3, K, K), generator=g, device="cuda") * 0.1
    d = L.desc(2, 3, 3, 70, W, K, 3, L.GIGA_BORDER_CLAMP if border == "clamp" else 0,
               giga.DTYPES[dtype], 0)
    n = x.numel()
    for choice in range(8):  # each forward candidate; fused, two-pass and ring backward
        L.check(L.giga_autotune_set_choice(d, 1, choice), "pin")
        L.check(L.giga_autotune_set_choice(d, 2, choice), "pin")
        L.check(L.giga_autotune_set_choice(d, 6, (0, 1, 5, 6)[choice % 4]), "pin")
        y0, dx0 = giga.conv2d_fwd(x, w, border), giga.conv2d_bwd_input(dy, w, border)
        both0 = giga.conv2d_bwd(x, dy, w, border)
        for ref, call in (
                (y0, lambda out: giga.conv2d_fwd(x, w, border, out=out)),
                (dx0, lambda out: giga.conv2d_bwd_input(dy, w, border, out=out)),
                (both0[0], lambda out: dws.append(giga.conv2d_bwd(x, dy, w, border, dx=out)[1]))):
            dws = []
            out, buf = hole(shape, dtype, offset)
            call(out)
            assert torch.equal(out, ref) and untouched(buf, offset, n), choice
            assert all(torch.equal(dw, both0[1]) for dw in dws), choice
    L.giga_autotune_clear()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("W,offset", [(8, 1), (136, 3), (392, 2)])
def test_separable_and_gray(giga, dtype, W, offset):
    x = torch.rand((2, 3, 70, W), device="cuda").to(dtype)
    for border in ("zero", "clamp"):
        for K in (1, 3, 9, 13, 15, 31):
            f = torch.rand((3, K), device="cuda")
            out, buf = hole(x.shape, dtype, offset)
            giga.conv2d_separable(x, f, f, border, out=out)
            assert torch.equal(out, giga.conv2d_separable(x, f, f, border))
            assert untouched(buf, offset, x.numel())
        for K in (1, 3, 7, 15):
            w = torch.rand((1, K, K), device="cuda")
            out, buf = hole((2, 1, 70, W), dtype, offset)
            giga.gray_conv2d(x, w, border, out=out)
            assert torch.equal(out, giga.gray_conv2d(x, w, border))
            assert untouched(buf, offset, out.numel())
