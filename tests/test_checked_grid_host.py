"""The grid of passes whose tables are checked for flip symmetry on the device: an
instance that turns out not to be symmetric has all of its tiles, and gets a CTA for
each while the batch has no more tiles than the device SMs."""
import ctypes

import pytest

from paper_2401_02852_gb300 import _lib


def _grid(name, batch, tiles, *slots):
    f = _lib.load()[f"_ZN4qaoa{len(name)}{name}E{'i' * len(slots)}im"]
    return f(*(ctypes.c_int(s) for s in slots), ctypes.c_int(batch), ctypes.c_uint64(tiles))


@pytest.mark.parametrize("per", [1, 2])  # resident CTAs per SM
@pytest.mark.parametrize("batch", [1, 3, 8, 76, 152, 300, 5000])
@pytest.mark.parametrize("bits", range(1, 18))
def test_width(per, batch, bits):
    sms, tiles = 152, 1 << bits
    slots = sms * per
    gx = _grid("checked_grid_x", batch, tiles, sms, slots)
    if batch * tiles <= sms:
        assert gx == tiles
    else:
        assert gx == _grid("balanced_grid_x", batch, tiles // 2, slots) and 1 <= gx <= slots
