"""The pyramid kernel's threads cover a frame's chunks once, also in frames wider than the detector takes (the tracker
takes any width): the device code's own index arithmetic, compiled for the host."""
import ctypes

import numpy as np
import pytest

from test_host_order import host_lib  # noqa: F401


# 2^16 chunks of 16 columns per row and around it, and the widest frame that a tracker accepts
@pytest.mark.parametrize("w,h", [(7, 7), (31, 40), (752, 480), (65535, 300), (1048576, 30), (1048577, 30),
                                 (1052688, 40), (2097169, 28), (16000033, 16), (38347919, 7)])
@pytest.mark.parametrize("levels", [1, 3])
def test_every_chunk_once(host_lib, w, h, levels):  # noqa: F811
    if h >> (levels - 1) < 7:
        pytest.skip("smaller than the pyramid allows")
    cx, rows = max(2, -(-w // 16)), 4 if levels == 1 else 1 << (levels - 1)
    n_chunks = cx * -(-h // rows)
    blocks = host_lib.fake_pyramid_chunks(w, h, levels, 0, 0, None)
    assert blocks == -(-n_chunks // 256)
    # blocks at the start, at the end, and where rows of chunks begin
    pick = {0, blocks - 1} | {r * cx // 256 + d for r in range(-(-h // rows)) for d in (-1, 0, 1)}
    for b in sorted(b for b in pick if 0 <= b < blocks):
        out = np.zeros((256, 2), np.int32)
        host_lib.fake_pyramid_chunks(w, h, levels, b, 1, ctypes.c_void_p(out.ctypes.data))
        chunk = b * 256 + np.arange(256)
        assert np.array_equal(out[:, 0], chunk % cx) and np.array_equal(out[:, 1], chunk // cx), b
