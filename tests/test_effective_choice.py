"""giga_autotune_effective_choice: the configuration a call takes, whether stored
or picked by the built-in rule (giga_autotune_choice says 0 both for a stored 0
and for none).  No GPU: sizes far from every threshold of the rule."""
import pytest

from paper_2504_01266_gb300 import _lib as L

FWD, BOTH = 1, 6


@pytest.fixture()
def lib():
    from paper_2504_01266_gb300 import build
    build.build()
    mode = L.giga_autotune_get_mode()
    L.giga_autotune_clear()
    L.giga_autotune_set_mode(1)
    yield L
    L.giga_autotune_clear()
    L.giga_autotune_set_mode(mode)


def desc(N, side, K, dtype=0, W=None):
    return L.desc(N, 3, 3, side, W or side, K, 3, 0, dtype, L.GIGA_LAYOUT_NCHW)


@pytest.mark.parametrize("args,op,want", [
    ((1, 64, 7), FWD, 1), ((1, 512, 21), FWD, 1), ((1, 512, 31), FWD, 0), ((1, 64, 31), FWD, 1),
    ((2, 512, 31), FWD, 1), ((16, 2048, 7), FWD, 4), ((16, 2048, 5), FWD, 0),
    ((16, 2048, 3, 1), FWD, 4), ((16, 2048, 3, 1, 2046), FWD, 0),
    ((1, 64, 3), BOTH, 0), ((4, 2048, 3), BOTH, 6), ((64, 2048, 3), BOTH, 1),
    ((4, 2048, 3, 0, 2046), BOTH, 0), ((16, 2048, 15), BOTH, 5), ((16, 2048, 7), BOTH, 0),
    ((16, 2048, 7, 1), BOTH, 5), ((16, 2048, 7), 4, 0), ((16, 2048, 7), 2, 4)])
def test_rule(lib, args, op, want):
    d = desc(*args)
    assert L.giga_autotune_effective_choice(d, op) == want
    assert L.giga_autotune_choice(d, op) == 0  # nothing stored
    for pin in (0, 3):
        assert L.giga_autotune_set_choice(d, op, pin) == L.GIGA_OK
        assert L.giga_autotune_effective_choice(d, op) == pin
    L.giga_autotune_set_mode(0)  # stored choices are not used
    assert L.giga_autotune_effective_choice(d, op) == want


def test_errors(lib):
    d = desc(1, 64, 7)
    assert L.giga_autotune_effective_choice(d, 3) == -1
    d.K = 4
    assert L.giga_autotune_effective_choice(d, FWD) == -1
