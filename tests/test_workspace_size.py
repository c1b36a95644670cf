"""The instance-sized part of a workspace (gs_workspace_size, host only): each eye's
buffers follow that eye's own capacity.

Per instance of an eye: surfel id 4 B, span 4 B, row-list entry 4 B, and for the first
eight per surfel the second ranges' 8 B and their row-list entries' 4 B.
"""
import ctypes as C

import pytest

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gs():
    from paper_2609_30741_gb300 import build
    build.build()
    from paper_2609_30741_gb300 import gs as gsmod
    return gsmod


def _size(gs, n, cap, cap_aff):
    lim = gs.Limits(n, 640, 480, cap, 1024, 0, 16, 0, cap_aff, 0)
    out = C.c_size_t()
    assert gs.lib().gs_workspace_size(C.byref(lim), C.byref(out)) == gs.GS_OK
    return out.value


def _eye(n, cap):
    return 12 * cap + 12 * min(cap, 8 * n)


@pytest.mark.parametrize("n,cap", [(20000, 1 << 21), (3000000, 1 << 27), (3000000, 1 << 28), (500000, 48000000)])
def test_a_small_eye_takes_little_beside_a_large_one(gs, n, cap):
    small = 1 << 16
    base = _size(gs, n, small, small)
    tol = 256 * 8
    assert abs(_size(gs, n, cap, small) - base - (_eye(n, cap) - _eye(n, small))) <= tol
    assert abs(_size(gs, n, small, cap) - base - (_eye(n, cap) - _eye(n, small))) <= tol
    assert abs(_size(gs, n, cap, 0) - base - 2 * (_eye(n, cap) - _eye(n, small))) <= tol
