"""vio_get_tuning tells a call of the tile kernel, which is no built variant, from a persistent launch (host code over
the fake CUDA runtime, whose kernels fit four to an SM)."""
import ctypes

import pytest

from paper_2003_13493_gb300 import vio
from test_host_order import S1, host, host_lib  # noqa: F401


def tuning(h):
    t = vio.Tuning()
    assert h.lib.vio_get_tuning(h.ctx, ctypes.byref(t)) == 0
    return {name: getattr(t, name) for name, _ in vio.Tuning._fields_}


# one frame: tiles of 32 score rows; 12 frames: of 64
@pytest.mark.parametrize("n,rows", [(1, 32), (12, 64)])
@pytest.mark.parametrize("radius", [1, 3])
def test_tile_calls_are_reported_as_such(host, n, rows, radius):  # noqa: F811
    sizes = [(640, 480)] * n
    h = host(max_frames=64, nms_radius=radius)
    first = vio.variant_ids(radius)[0]
    tw, th, _ = vio.variants()[first]
    assert h.detect(sizes, S1, cell=64) == 0
    t = tuning(h)
    # no count of persistent CTAs was launched; the tile is the kernel's own
    assert (t["cta_per_sm"], t["tile_w"], t["tile_h"]) == (0, 120, rows - 2 * radius)
    assert (t["variant"], t["nms_radius"], t["cell_size"]) == (first, radius, 64)
    # pinning what was reported gives the variant's persistent launch, as many CTAs as fit
    pin = vio.Tuning(0, 0, t["cta_per_sm"], t["variant"], 0, 0)
    assert h.lib.vio_set_tuning(h.ctx, ctypes.byref(pin)) == 0
    assert h.detect(sizes, S1, cell=64) == 0
    assert tuning(h) == dict(t, cta_per_sm=4, tile_w=tw, tile_h=th)
    assert h.lib.vio_set_tuning(h.ctx, None) == 0
    assert h.detect(sizes, S1, cell=64) == 0
    assert tuning(h) == t
    # calls that the tile kernel does not take
    assert h.sweep(sizes, S1) == 0
    assert tuning(h)["cta_per_sm"] == 4 and tuning(h)["tile_h"] == th
    assert h.detect([(1920, 1080)] * 60, S1) == 0
    assert tuning(h)["cta_per_sm"] == 4 and tuning(h)["tile_h"] == th
