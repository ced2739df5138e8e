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


def _room(gib):
    if torch.cuda.mem_get_info()[0] < gib * 2 ** 30:
        pytest.skip(f"needs {gib} GiB of device memory")


@pytest.mark.parametrize("case", ["one bin", "ramp"])
def test_map_of_frames_beyond_32_bit_counts(g, case):
    """One bin that holds more than 2^32 pixels; a ramp with more than 2^32 pixels in the bins below the middle's."""
    _room(60)
    if case == "one bin":
        n = 65600
        ref = torch.full((n, n), 2.5, device="cuda")
        ref[5] = 3.5
        want = np.arange(n) == 5
    else:
        n = 100000
        ref = torch.arange(n, dtype=torch.float32, device="cuda")[:, None].expand(n, n).contiguous()
        # n values of each row number: median (n - 1) / 2, sigma sqrt((n^2 - 1) / 12)
        want = np.abs(np.arange(n) - (n - 1) / 2) > np.sqrt((n * n - 1.0) / 12.0)
    got = g.context().graphic_bad_pixel_map(ref, 1.0)
    lo, hi = got.amin(dim=1).cpu().numpy(), got.amax(dim=1).cpu().numpy()
    assert np.array_equal(lo, want) and np.array_equal(hi, want)
    del ref, got
    torch.cuda.empty_cache()


def test_correction_of_a_frame_of_2_32_bad_pixels(g):
    _room(60)
    n = 65536
    ctx = g.Context(torch.cuda.current_device())   # its scratch, as large as the frame, goes with it
    try:
        x = torch.full((1, n, n), float("nan"), device="cuda")
        ctx._stream()
        rc = g.lib().graphic_bad_pixel_fix(ctx.h, ctypes.c_void_p(x.data_ptr()), 1, n, None)
        assert rc == -5, rc
        x.fill_(2.0)
        x[0, 7, 9] = float("inf")
        rc = g.lib().graphic_bad_pixel_fix(ctx.h, ctypes.c_void_p(x.data_ptr()), 1, n, None)
        assert rc == 0, rc
        assert bool((x == 2.0).all())
        del x
    finally:
        ctx.close()
    torch.cuda.empty_cache()
