"""Workspace sizes follow from the arguments alone: a host without a GPU, or a program that has not chosen its
device yet, gets the size that the call asks for later (CPU)."""
import ctypes

import pytest

from paper_2408_03538_gb300 import _lib as L


def _up(x):
    return (x + 255) // 256 * 256


@pytest.mark.parametrize("n,S", [(1, 1), (300, 7), (100_000, 128), (300_001, 256)])
def test_transfer_backward_size_does_not_depend_on_the_device(n, S):
    p = L.TransferParams(3, S, None, 0.0, 1.0, L.SHADOW, 0, None)
    got = L.load().prtgs_transfer_backward_workspace_size(n, ctypes.byref(p))
    batch = min(n, max(2**26 // S // 64 * 64, 64))
    blocks = min(152 * 4, max(1, (8 * -(-batch // 256) * S + 3) // 4))  # 4 per SM, or a warp per packet
    assert got == 256 + 2 * _up(4 * batch * S) + _up(96 * n) + _up(4 * blocks * 4 * 2048)
