"""The training step's scratch (gs_repair_train_scratch_size, host only) is what a tile
keeps, six layers' inputs, the raw outputs, two gradients and its statistics, and beside
it the partial gradients of the last layer, 4.6 KB for each multiprocessor (152 assumed
without a GPU).
"""
import ctypes as C

import pytest

torch = pytest.importorskip("torch")

TILE = 6 * 4 * 832 * 16 + 4 * 256 * 4 + 4 + 2 * 4 * 832 * 16 + 32


@pytest.mark.parametrize("n", [1, 64, 512, 5000])
def test_scratch_is_the_tiles_own(n):
    from paper_2609_30741_gb300 import build
    build.build()
    from paper_2609_30741_gb300 import gs
    size = C.c_size_t()
    assert gs.lib().gs_repair_train_scratch_size(n, C.byref(size)) == gs.GS_OK
    assert 0 < size.value - n * TILE <= min(n, 160) * 4 * (4 * 9 * 32 + 4) + 4096
