"""The built-in choice goes by what TMA can load: BF16 planes whose base is 8 but
not 16 bytes aligned take the same kernels as planes with odd rows, not those
chosen for aligned ones."""
import pytest
import torch

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
    _lib.giga_autotune_set_mode(mode)


def kernels(call):
    """Names of the kernels that `call` launches (the profiler's first session of
    a process may come back empty)."""
    names = ""
    for _ in range(5):
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            call()
            torch.cuda.synchronize()
        names = " ".join(e.name for e in prof.events() if "giga" in e.name)
        if names:
            break
    return names


@pytest.mark.parametrize("K,per_sm,aligned_kernel", [(3, 4, "dw_bwd_ring_kernel"),
                                                     (9, 4, "dw_filter_kernel")])
def test_bf16_base(giga, K, per_sm, aligned_kernel):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    shape = (per_sm * sms, 1, 16, 128)
    n = per_sm * sms * 16 * 128
    w = torch.zeros((1, K, K), device="cuda")
    names = {}
    for offset in (0, 4):
        x, dy, dx = (torch.zeros(n + 8, dtype=torch.bfloat16, device="cuda")[offset:offset + n]
                     .view(shape) for _ in range(3))
        names[offset] = kernels(lambda: giga.conv2d_bwd(x, dy, w, dx=dx))
    assert aligned_kernel in names[0], names
    assert aligned_kernel not in names[4] and "dw_bwd_kernel" in names[4], names
