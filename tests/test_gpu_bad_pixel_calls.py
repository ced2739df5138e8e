"""Bad pixel map and correction where a call is refused, where a frame holds
more than 2^32 pixels, and where frames change from the listed fill to the
dense passes."""
import ctypes

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    from paper_1510_04331_gb300 import graphic
    return graphic


@pytest.mark.parametrize("n", [7, 256])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_map_of_a_refused_frame_is_left_alone(g, n, value):
    ref = torch.randn((n, n), device="cuda")
    ref[n // 2, n - 1] = float(value)
    bad = torch.full((n, n), 7, dtype=torch.uint8, device="cuda")
    ctx = g.context()
    ctx._stream()
    rc = g.lib().graphic_bad_pixel_map(ctx.h, ctypes.c_void_p(ref.data_ptr()), n, 2.0, ctypes.c_void_p(bad.data_ptr()))
    assert rc == -5, rc
    assert bool((bad == 7).all())
